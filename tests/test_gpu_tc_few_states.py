"""States are filtered independently: a block's first n states give the same bits
whatever else the block holds. n runs over the edges of the one- and two-tile
units (128 states), for every unit shape and accumulator width; the two-tile
kernels are also compared with the FP64 oracle there."""
import numpy as np
import pytest
import torch

from oracle import chefsi as O
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu

SHAPES = {32: [(4, 2, 0), (2, 2, 0), (4, 2, 1), (4, 2, 2)],
          64: [(2, 2, 0), (1, 2, 0), (2, 1, 0), (2, 2, 1), (2, 2, 2)],
          128: [(2, 1, 0), (1, 2, 0), (1, 2, 1), (1, 2, 2)]}
U_OP = {"tf32": 2.0 ** -9, "bf16": 2.0 ** -8, "bf16x3": 2.0 ** -16}


@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
@pytest.mark.parametrize("nb,acc", [((9, 32), 32), ((33, 64), 64), ((40, 120), 128)])
def test_first_states_do_not_depend_on_the_rest(prec, nb, acc):
    cfg = G.ProblemConfig(name="few", grid=(3, 3, 2), periodic=(True, True, False), stencil="27", nb=nb, Ns=260, m=4,
                          Ne=1.0, seed=8)
    H = G.make_blocks(cfg)
    X = np.random.default_rng(9).standard_normal((260, H.N))
    a0, a, b = -1.8, 3.0, 46.0
    ref = O.chebyshev_filter(O.DGHamiltonian.from_blocksparse(H), X.T, cfg.m, a, b, a0).T
    with D.Context(H) as ctx:
        Xd = torch.from_numpy(X).cuda()
        for G_, T, lay in SHAPES[acc]:
            ctx.set_tile_shape(prec, G_, T, lay)
            full = ctx.filter(Xd, cfg.m, a, b, a0, prec=prec)
            err = np.linalg.norm(full.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= 2 * cfg.m * U_OP[prec], (G_, T, lay, err)
            for n in (1, 127, 128, 129, 256):
                part = ctx.filter(Xd[:n].contiguous(), cfg.m, a, b, a0, prec=prec)
                assert torch.equal(part, full[:n]), (G_, T, lay, n)
            g = ctx.filter_graph(Xd[:100].contiguous(), cfg.m, a, b, a0, prec=prec)
            assert torch.equal(g, full[:100]), (G_, T, lay)
