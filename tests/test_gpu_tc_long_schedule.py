"""Filters of up to 128 states whose group schedule fits shared memory beside the
two-tile kernel's ring but not beside the larger one-tile ring: one element
coupled to every other one, around the lengths at which either ring stops
fitting, and on both sides of 128 states."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu
U_OP = {"tf32": 2.0 ** -9, "bf16x3": 2.0 ** -16}  # of a product, as in test_gpu_tc.py


def star(M, seed=1):
    """Element 0 coupled to all others, those to it and themselves; sizes 1..3."""
    rng = np.random.default_rng(seed)
    nb = (1 + np.arange(M) % 3).astype(np.int32)
    row_ptr = np.concatenate([[0], M + 2 * np.arange(M)])
    col, off, vals, at = [], [], [], 0
    arm = [None] + [0.01 * rng.standard_normal((nb[0], nb[K])) for K in range(1, M)]

    def put(c, block):
        nonlocal at
        col.append(c)
        off.append(at)
        vals.append(np.ascontiguousarray(block).ravel())
        at += block.size

    def diagonal(K):
        a = rng.standard_normal((nb[K], nb[K]))
        return 0.1 * (a + a.T) + np.diag(rng.uniform(0.0, 40.0, nb[K]))

    put(0, diagonal(0))
    for K in range(1, M):
        put(K, arm[K])
    for K in range(1, M):
        put(0, arm[K].T)
        put(K, diagonal(K))
    return G.BlockSparse(nb=nb, row_ptr=row_ptr.astype(np.int64), col=np.array(col, dtype=np.int32),
                         blk_off=np.array(off, dtype=np.int64), values=np.concatenate(vals))


@pytest.mark.parametrize("M", [1350, 1450, 2700])
@pytest.mark.parametrize("prec", ["tf32", "bf16x3"])
def test_every_state_count_is_accepted(M, prec):
    """The states of every count are those of the largest one to the bit (one shape,
    chosen at the first call), and that is within 2 m u_op of the FP64 filter."""
    H = star(M)
    m, a, b, a0 = 4, 5.0, 45.0, -2.0
    X = torch.from_numpy(np.random.default_rng(2).standard_normal((129, H.N))).cuda()
    with D.Context(H) as ctx:
        first = ctx.filter(X[:16].contiguous(), m, a, b, a0, prec=prec)
        Y = ctx.filter(X, m, a, b, a0, prec=prec)
        Z = ctx.filter(X, m, a, b, a0, prec="f64")
        assert float((Y - Z).norm()) <= 2 * m * U_OP[prec] * float(Z.norm())
        assert torch.equal(first, Y[:16])
        for Ns in (128, 48):
            part = X[:Ns].contiguous()
            assert torch.equal(ctx.filter(part, m, a, b, a0, prec=prec), Y[:Ns])
            assert torch.equal(ctx.filter_graph(part, m, a, b, a0, prec=prec), Y[:Ns])
