"""The buffer of partial sums of the split FP64 products is optional: without the
memory for it, and under a stream capture, the calls succeed with the bits they
have with it."""
import numpy as np
import pytest
import torch

import fake_cuda_malloc
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def test_calls_without_the_memory_for_parts(tmp_path):
    fake_cuda_malloc.run(tmp_path, r"""
from paper_1606_03416_gb300.autograd import band_energy
cfg = G.ProblemConfig(name="oom", grid=(3, 3, 2), periodic=(True, True, True), stencil="27", nb=40, Ns=200, m=6,
                      Ne=300.0, seed=2, scales={1: 0.05, 2: 0.02, 3: 0.01})
H = G.make_blocks(cfg)
rng = np.random.default_rng(3)
X = torch.from_numpy(rng.standard_normal((200, H.N))).cuda()
f = torch.from_numpy(rng.uniform(0.0, 1.0, 200)).cuda()
v = torch.from_numpy(rng.standard_normal(H.N)).cuda()
P128 = 128 << 20
def results(products):
    with D.Context(H) as ctx:
        ctx.set_subspace_products(products)
        Y = X.clone()
        out = ctx.cycle(Y, 6, 300.0, 0.05, v0=v)
        Z = X.clone()
        ritz = ctx.rayleigh_ritz(Z)
        E, _, Hb, Xb = ctx.energy_grad(X, 4, 10.0, 45.0, -1.7, 300.0, 0.05)
        return [ctx.gram(X), ctx.density_blocks(X, f), Y, out["ritz"], out["P"], Z, ritz, Hb, Xb,
                torch.tensor(E)]
for products in ("f64", "sliced_bf16"):
    want = results(products)
    deny(P128, P128)
    got = results(products)
    deny(1, 0)
    for a, b in zip(want, got):
        assert torch.equal(a, b), products
""")


@pytest.mark.parametrize("nb,Ns", [(40, 200), ((17, 90), 700), (4, 3)])
def test_first_calls_under_capture(nb, Ns):
    """On a context that has run nothing, and again after eager calls."""
    cfg = G.ProblemConfig(name="cap", grid=(4, 3, 2), periodic=(True, True, True), stencil="27", nb=nb, Ns=Ns, m=2,
                          Ne=1.0, seed=8)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(9)
    X = torch.from_numpy(rng.standard_normal((Ns, H.N))).cuda()
    f = torch.from_numpy(rng.uniform(0.0, 1.0, Ns)).cuda()
    with D.Context(H) as ctx, D.Context(H) as fresh:
        S0, P0 = ctx.gram(X), ctx.density_blocks(X, f)
        for c in (fresh, ctx):
            S, P = torch.zeros_like(S0), torch.zeros_like(P0)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                c.gram(X, S)
                c.density_blocks(X, f, P)
            for _ in range(2):
                g.replay()
            torch.cuda.synchronize()
            assert torch.equal(S, S0) and torch.equal(P, P0)
