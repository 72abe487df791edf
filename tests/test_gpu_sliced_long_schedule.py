"""The sliced H X on patterns whose groups of elements couple to more slices than
the pair kernel's shared memory holds: small elements with some hundred random
neighbours, on both sides of that length, and one element coupled to all others.
Integer H and states: the bits of the FP64 product."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def random_pattern(M, chance, hub, nb, seed=1):
    """Elements of nb functions; a pair couples with this chance, element 0 (hub) with every other one."""
    rng = np.random.default_rng(seed)
    C = np.triu(rng.random((M, M)) < chance, 1)
    C[0, 1:] |= hub
    C = C | C.T | np.eye(M, dtype=bool)
    row_ptr = np.concatenate([[0], np.cumsum(C.sum(1))]).astype(np.int64)
    col = np.nonzero(C)[1].astype(np.int32)
    row = np.repeat(np.arange(M), np.diff(row_ptr))
    off = np.arange(len(col), dtype=np.int64) * nb * nb
    vals = rng.integers(-50, 50, size=(len(col), nb, nb)).astype(np.float64)
    at = np.full((M, M), -1)
    at[row, col] = np.arange(len(col))
    lower = np.nonzero(row > col)[0]
    vals[lower] = vals[at[col[lower], row[lower]]].transpose(0, 2, 1)
    diag = at[np.arange(M), np.arange(M)]
    vals[diag] += vals[diag].transpose(0, 2, 1).copy()
    return G.BlockSparse(nb=np.full(M, nb, dtype=np.int32), row_ptr=row_ptr, col=col, blk_off=off, values=vals.ravel())


@pytest.mark.parametrize("M,chance,hub,nb", [(300, 0.3, False, 2), (1200, 0.23, False, 1), (1200, 0.23, True, 3),
                                             (3000, 0.0, True, 1)])
def test_matches_the_fp64_product(M, chance, hub, nb):
    H = random_pattern(M, chance, hub, nb)
    X = torch.from_numpy(np.random.default_rng(2).integers(-1000, 1000, size=(70, H.N)).astype(np.float64)).cuda()
    with D.Context(H) as ctx:
        assert torch.equal(ctx.sliced_matvec(X), ctx.matvec(X))
