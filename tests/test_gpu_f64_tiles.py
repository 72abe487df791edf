"""The FP64 tiles at their edges: element sizes around the 8- and 64-column and
4- and 16-row groups, states around the 16-row tile, products split into parts
(few states, many rows) and not, on strided blocks. Against the oracle's
arithmetic in NumPy, at K u times the sum of magnitudes."""
import numpy as np
import pytest
import torch

from oracle import chefsi as O
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def strided(a, pad=3):
    big = torch.full((a.shape[0], a.shape[1] + pad), 7.0, dtype=torch.float64, device="cuda")
    big[:, :a.shape[1]] = torch.from_numpy(a).cuda()
    return big[:, :a.shape[1]]


@pytest.mark.parametrize("nb", [1, 8, (7, 9), (15, 17), 40, (63, 66), (120, 130), 256])
@pytest.mark.parametrize("Ns", [1, 15, 17, 65])
def test_element_products_at_tile_edges(nb, Ns):
    cfg = G.ProblemConfig(name="edge", grid=(3, 2, 1), periodic=(True, True, False), stencil="9", nb=nb, Ns=Ns, m=2,
                          Ne=1.0, seed=3, scales={1: 0.05, 2: 0.02})
    H = G.make_blocks(cfg)
    Ho = O.DGHamiltonian.from_blocksparse(H)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((Ns, H.N))
    f = rng.uniform(0.0, 1.0, Ns)
    off = np.concatenate([[0], np.cumsum(H.nb)])
    with D.Context(H) as ctx:
        Xd, fd = strided(X), torch.from_numpy(f).cuda()
        Y = ctx.matvec(Xd, strided(np.zeros_like(X))).cpu().numpy()
        P = ctx.unpack_density(ctx.density_blocks(Xd, fd))
        Q = ctx.density_pattern(Xd, fd).cpu().numpy()
        S = ctx.gram(Xd).cpu().numpy()
    absH = H.values.copy()
    Ha = G.BlockSparse(nb=H.nb, row_ptr=H.row_ptr, col=H.col, blk_off=H.blk_off, values=np.abs(absH))
    mag = O.matvec(O.DGHamiltonian.from_blocksparse(Ha), np.abs(X).T).T
    assert np.all(np.abs(Y - O.matvec(Ho, X.T).T) <= 4 * 9 * 256 * U * mag)
    for K in range(H.M):
        x = X[:, off[K]:off[K + 1]]
        ref, a = x.T @ (f[:, None] * x), np.abs(x).T @ (f[:, None] * np.abs(x))
        got = P[K].cpu().numpy()
        assert np.all(np.abs(got - ref) <= 4 * (Ns + 2) * U * a + 1e-300)
        assert np.array_equal(got, got.T)
        for e in range(H.row_ptr[K], H.row_ptr[K + 1]):
            y = X[:, off[H.col[e]]:off[H.col[e] + 1]]
            ref, a = x.T @ (f[:, None] * y), np.abs(x).T @ (f[:, None] * np.abs(y))
            blk = Q[H.blk_off[e]:H.blk_off[e] + ref.size].reshape(ref.shape)
            assert np.all(np.abs(blk - ref) <= 4 * (Ns + 2) * U * a + 1e-300)
    assert np.all(np.abs(S - X @ X.T) <= 4 * H.N * U * (np.abs(X) @ np.abs(X).T))
    assert np.array_equal(S, S.T)


@pytest.mark.parametrize("Ns", [2, 16, 100, 333, 700])
def test_gram_and_density_in_parts(Ns):
    """Few tiles and long sums (split into parts) up to enough tiles for the
    whole GPU; densities of few elements and many states."""
    cfg = G.ProblemConfig(name="parts", grid=(4, 4, 2), periodic=(True, True, True), stencil="27", nb=(40, 72), Ns=Ns,
                          m=2, Ne=1.0, seed=5)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(6)
    X = rng.standard_normal((Ns, H.N))
    f = rng.uniform(0.0, 1.0, Ns)
    off = np.concatenate([[0], np.cumsum(H.nb)])
    with D.Context(H) as ctx:
        Xd = torch.from_numpy(X).cuda()
        S = ctx.gram(Xd).cpu().numpy()
        P = ctx.unpack_density(ctx.density_blocks(Xd, torch.from_numpy(f).cuda()))
    assert np.all(np.abs(S - X @ X.T) <= 4 * H.N * U * (np.abs(X) @ np.abs(X).T))
    assert np.array_equal(S, S.T)
    for K in range(H.M):
        x = X[:, off[K]:off[K + 1]]
        ref, a = x.T @ (f[:, None] * x), np.abs(x).T @ (f[:, None] * np.abs(x))
        assert np.all(np.abs(P[K].cpu().numpy() - ref) <= 4 * (Ns + 2) * U * a)
