"""New values of H give back large buffers of the sliced H X (1.5 GB here) and keep
small ones; the product afterwards has the bits of a new context."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("grid,nb,Ns,given_back", [((6, 6, 6), 64, 2000, True), ((3, 3, 3), 40, 300, False)])
def test_large_buffers_are_given_back(grid, nb, Ns, given_back):
    cfg = G.scaled_copy(G.CONFIGS["bulk3d_8x8x8"], grid=grid, nb=nb, Ns=Ns)
    H = G.make_blocks(cfg)
    X = torch.from_numpy(np.random.default_rng(1).standard_normal((Ns, H.N))).cuda()
    vals = torch.from_numpy(H.values).cuda()
    Y, Z = torch.empty_like(X), torch.empty_like(X)
    with D.Context(H) as ctx, D.Context(H) as new:
        ctx.set_values(2 * vals)
        before = free_bytes()
        ctx.sliced_matvec(X, Y)
        used = before - free_bytes()
        ctx.set_values(vals)
        kept = before - free_bytes()
        # digits of H (7 x 2 bytes an entry of 64-wide slices), of the states, and 7 slabs of INT32
        if given_back:
            big = 14 * int(H.row_ptr[-1]) * 64 * 64 + (14 + 28) * Ns * H.N
            assert big > 1.4e9 and used >= big and kept <= used - big
        else:
            assert kept == used
        assert torch.equal(ctx.sliced_matvec(X, Y), new.sliced_matvec(X, Z))
