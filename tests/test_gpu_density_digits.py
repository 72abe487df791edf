"""The cycle's density blocks from digits against density_blocks (FP64) of the
same states: sizes on both sides of the rule, elements that fill a 256-row tile
unevenly, several K chunks, one element per tile and many."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,nb,Ns", [((3, 3, 3), 40, 200), ((4, 4, 4), (17, 63), 1201), ((6, 5, 1), (40, 120), 1203),
                                        ((4, 3, 1), (129, 140), 1500), ((6, 6, 4), 33, 4099)])
def test_cycle_density_matches_fp64(grid, nb, Ns):
    """Either form is within (Ns + 8) u of sum_i f_i |x_ij x_ij'| <=
    sqrt(P_jj P_j'j') (u = 2^-53: Ns roundings of the FP64 sum and two of each
    term; the digits' form rounds sqrt(f) x twice in each factor and the sum
    once a chunk). P is symmetric to the bit."""
    cfg = G.scaled_copy(G.CONFIGS["bulk3d_8x8x8" if grid[2] > 1 else "sheet2d_24x20"], grid=grid, nb=nb, Ns=Ns)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(4)
    with D.Context(H) as ctx:
        ctx.set_subspace_products("sliced_bf16", 10)
        X = torch.from_numpy(rng.standard_normal((Ns, H.N))).cuda()
        out = ctx.cycle(X, m=4, Ne=1.1 * Ns, kT=0.05, v0=torch.from_numpy(rng.standard_normal(H.N)).cuda(), prec="f64")
        P = ctx.unpack_density(out["P"])
        Q = ctx.unpack_density(ctx.density_blocks(X, out["f"]))
        for p, q in zip(P, Q):
            p, q = p.cpu().numpy(), q.cpu().numpy()
            d = np.sqrt(np.diag(q))
            assert np.array_equal(p, p.T)
            assert (np.abs(p - q) <= 2 * (Ns + 8) * 2.0 ** -53 * np.outer(d, d)).all()
