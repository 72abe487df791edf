"""The Lanczos bound in one launch and the Fermi level on a cluster, at the
edges of how they split their work: few and many rows, more than 32 neighbour
blocks in a row, elements of more than 64 functions, an invariant start vector;
one state up to several per thread."""
import numpy as np
import pytest
import torch

from oracle import chefsi as O
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def all_coupled(nb, seed=0):
    """Every element couples to every other one (row_ptr of len(nb) blocks)."""
    rng = np.random.default_rng(seed)
    nb = np.asarray(nb, dtype=np.int32)
    off = np.concatenate([[0], np.cumsum(nb)])
    A = rng.standard_normal((off[-1], off[-1]))
    A = 0.05 * (A + A.T) + np.diag(rng.uniform(-1.0, 40.0, off[-1]))
    vals, offs, pos = [], [], 0
    for K in range(nb.size):
        for L in range(nb.size):
            offs.append(pos)
            vals.append(A[off[K]:off[K + 1], off[L]:off[L + 1]].ravel())
            pos += vals[-1].size
    M = nb.size
    return G.BlockSparse(nb=nb, row_ptr=np.arange(M + 1, dtype=np.int64) * M,
                         col=np.tile(np.arange(M, dtype=np.int32), M), blk_off=np.asarray(offs, dtype=np.int64),
                         values=np.concatenate(vals))


@pytest.mark.parametrize("nb,k", [([1], 1), ([3], 5), ([7] * 5, 10), ([5] * 33, 12), ([3, 70, 1, 130, 64, 65], 20),
                                  ([16] * 70, 64), ([256, 255, 33, 2], 9)])
def test_bounds_against_oracle(nb, k):
    H = all_coupled(nb, seed=len(nb))
    v = np.random.default_rng(3).standard_normal(H.N)
    b, t, _, _ = O.lanczos_bounds(O.DGHamiltonian.from_blocksparse(H), v, k)
    with D.Context(H) as ctx:
        got = ctx.bounds(torch.from_numpy(v).cuda(), k)
    scale = max(abs(b), abs(t))
    assert abs(got[0] - b) <= 1e-9 * scale and abs(got[1] - t) <= 1e-9 * scale


def test_bounds_stop_on_an_invariant_start_vector():
    H = all_coupled([4] * 3)
    H.values[:] = 0.0
    off = np.concatenate([[0], np.cumsum(H.nb)])
    for K in range(H.M):
        e = K * H.M + K
        H.values[H.blk_off[e]:H.blk_off[e] + 16] = np.diag(np.arange(off[K], off[K + 1]) + 1.0).ravel()
    v = np.zeros(H.N)
    v[4] = 2.5
    with D.Context(H) as ctx:
        b, t = ctx.bounds(torch.from_numpy(v).cuda(), 10)
        assert b == 5.0 and t == 5.0
        with pytest.raises(D.DGChefsiError):
            ctx.bounds(torch.full((H.N,), float("nan"), dtype=torch.float64, device="cuda"), 4)


@pytest.mark.parametrize("Ns", [1, 2, 255, 256, 257, 2047, 2049, 5000])
@pytest.mark.parametrize("kT,filling", [(0.01, 0.9), (0.3, 0.4), (1e-4, 0.97), (0.01, 0.0), (0.01, 1.0)])
def test_occupations_against_oracle(Ns, kT, filling):
    lam = np.sort(np.random.default_rng(Ns).uniform(-1.3, 2.0, Ns))
    Ne = 2.0 * round(filling * Ns)
    f, mu = O.fermi_occupations(lam, Ne, kT)
    with D.Context(all_coupled([2])) as ctx:
        got, m = ctx.occupations(torch.from_numpy(lam).cuda(), Ne, kT)
    got = got.cpu().numpy()
    assert abs(2 * got.sum() - Ne) <= 1e-12 * max(Ne, 1.0) + 1e-12
    # the level is where the count crosses N_e: its spread is that of the count's rounding over its slope
    slope = 2.0 * np.sum(f * (1.0 - f)) / kT
    if slope > 1e-6:
        assert abs(float(m) - mu) <= 1e-11 * max(Ne, 1.0) / slope + 1e-12
    assert np.max(np.abs(got - f)) <= 1e-9
