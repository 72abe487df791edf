"""The diagonal blocks of the pattern density equal density_blocks' bit for bit
and are symmetric: element sizes around a tile, sums split into parts and not,
strided states, and values stored with gaps and out of order."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def spread(H):
    """The same H with its blocks stored last to first, three doubles between them."""
    sizes = [int(H.nb[K]) * int(H.nb[H.col[e]]) for K in range(H.M) for e in range(H.row_ptr[K], H.row_ptr[K + 1])]
    off = np.zeros(len(sizes), dtype=np.int64)
    at = 3
    for e in reversed(range(len(sizes))):
        off[e] = at
        at += sizes[e] + 3
    values = np.zeros(at)
    for e, n in enumerate(sizes):
        values[off[e]:off[e] + n] = H.values[H.blk_off[e]:H.blk_off[e] + n]
    return G.BlockSparse(nb=H.nb, row_ptr=H.row_ptr, col=H.col, blk_off=off, values=values)


@pytest.mark.parametrize("moved", [False, True])
@pytest.mark.parametrize("nb,Ns", [(1, 1), (8, 700), ((15, 66), 333), (40, 64), ((120, 130), 130)])
def test_diagonal_blocks(nb, Ns, moved):
    cfg = G.ProblemConfig(name="pat", grid=(3, 3, 1), periodic=(True, True, False), stencil="9", nb=nb, Ns=Ns, m=2,
                          Ne=1.0, seed=3, scales={1: 0.05, 2: 0.02})
    H = G.make_blocks(cfg)
    if moved:
        H = spread(H)
    rng = np.random.default_rng(4)
    big = torch.from_numpy(rng.standard_normal((Ns, H.N + 3))).cuda()
    X, f = big[:, :H.N], torch.from_numpy(rng.uniform(0.0, 1.0, Ns)).cuda()
    with D.Context(H) as ctx:
        P = ctx.unpack_density(ctx.density_blocks(X, f))
        Q = ctx.density_pattern(X, f)
        Q2 = ctx.density_pattern(X, f, torch.full_like(Q, float("nan")))
    stored = torch.zeros_like(Q, dtype=torch.bool)
    for K in range(H.M):
        n = int(H.nb[K])
        for e in range(H.row_ptr[K], H.row_ptr[K + 1]):
            at, size = int(H.blk_off[e]), n * int(H.nb[H.col[e]])
            stored[at:at + size] = True
            if H.col[e] == K:
                q = Q[at:at + size].view(n, n)
                assert torch.equal(q, P[K]) and torch.equal(q, q.T)
    assert torch.equal(Q, Q2) and bool((Q[~stored] == 0).all())
