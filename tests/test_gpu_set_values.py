"""New values of H keep the sliced H X's layout and buffers: its results, the
filter's (direct and graph) and the reported unit shape are those of a context
made with the new values."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,nb,Ns,slices", [((3, 3, 2), 40, 70, (10, 10)), ((4, 4, 1), (40, 120), 300, (12, 10)),
                                               ((3, 2, 2), (17, 31), 33, (10, 12))])
def test_new_values_give_the_bits_of_a_new_context(grid, nb, Ns, slices):
    cfg = G.scaled_copy(G.CONFIGS["sheet2d_24x20" if grid[2] == 1 else "bulk3d_8x8x8"], grid=grid, nb=nb, Ns=Ns)
    H = G.make_blocks(cfg)
    X = torch.from_numpy(np.random.default_rng(1).standard_normal((Ns, H.N))).cuda()
    old = torch.from_numpy(H.values * 3.0).cuda()

    def results(ctx, s):
        return [ctx.sliced_matvec(X, slices=s), ctx.filter(X, 4, 5.0, 60.0, -2.0, prec="f64"),
                ctx.filter_graph(X, 4, 5.0, 60.0, -2.0, prec="f64").clone(), ctx.matvec(X)]

    with D.Context(H) as a, D.Context(H) as b:
        a.set_values(old)
        results(a, slices[0])
        a.filter(X, 4, 15.0, 180.0, -6.0, prec="bf16x3")
        a.set_values(torch.from_numpy(H.values).cuda())
        assert a.tile_shape("bf16x3")[:2] == b.tile_shape("bf16x3")[:2]
        for x, y in zip(results(a, slices[1]), results(b, slices[1])):
            assert torch.equal(x, y)
