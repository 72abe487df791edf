"""gram and density_blocks of one context on two streams at a time: both are
asynchronous and share the context's buffer of partial sums, and each result is
that of the call alone, to the bit."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def problem(nb, Ns, blocks):
    cfg = G.ProblemConfig(name="streams", grid=(4, 4, 4), periodic=(True, True, True), stencil="27", nb=nb, Ns=Ns, m=2,
                          Ne=1.0, seed=8)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(9)
    X = [torch.from_numpy(rng.standard_normal((Ns, H.N))).cuda() for _ in range(blocks)]
    f = [torch.from_numpy(rng.uniform(0.0, 1.0, Ns)).cuda() for _ in range(blocks)]
    return H, X, f


@pytest.mark.parametrize("nb,Ns", [(64, 300), ((17, 90), 1001)])
def test_two_streams_share_a_context(nb, Ns):
    H, X, f = problem(nb, Ns, 4)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    with D.Context(H) as ctx:
        S0 = [ctx.gram(x) for x in X]
        P0 = [ctx.density_blocks(x, g) for x, g in zip(X, f)]
        S = [torch.empty_like(s) for _ in range(5) for s in S0]
        P = [torch.empty_like(p) for _ in range(5) for p in P0]
        torch.cuda.synchronize()
        for k in range(len(S)):  # enqueued faster than they run, in turn on the two streams
            i = k % len(X)
            with torch.cuda.stream(streams[k % 2]):
                ctx.gram(X[i], S[k])
            with torch.cuda.stream(streams[(k + 1) % 2]):
                ctx.density_blocks(X[i], f[i], P[k])
        torch.cuda.synchronize()
        for k in range(len(S)):
            assert torch.equal(S[k], S0[k % len(X)]) and torch.equal(P[k], P0[k % len(X)])


def test_captured_after_an_eager_call():
    """A capture on one stream after eager calls on another, replayed: the graph
    waits for no event of theirs and shares no buffer with later calls."""
    H, X, f = problem(40, 200, 2)
    with D.Context(H) as ctx:
        S0, P0 = ctx.gram(X[0]), ctx.density_blocks(X[0], f[0])
        S, P = torch.zeros_like(S0), torch.zeros_like(P0)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.gram(X[0], S)
            ctx.density_blocks(X[0], f[0], P)
        for _ in range(3):
            g.replay()
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx.gram(X[1])
        torch.cuda.synchronize()
        # the same terms in another order: 2 N u (2 Ns u) times the sum of magnitudes
        u = 2.0 ** -53
        assert bool(((S - S0).abs() <= 2 * H.N * u * (X[0].abs() @ X[0].abs().T)).all())
        top = float(P0.abs().max())
        assert float((P - P0).abs().max()) <= 2 * 202 * u * top
