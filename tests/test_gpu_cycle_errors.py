"""A cycle that fails leaves its starting block as it was, also where the failure
is only seen after the eigensolve: H = c [[1, 1], [1, 1]] with c near the largest
double has finite entries and a finite H y, and its Ritz value 2 c is infinite."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def one_element(n, value):
    return G.BlockSparse(nb=np.array([n], dtype=np.int32), row_ptr=np.array([0, 1]), col=np.array([0], dtype=np.int32),
                         blk_off=np.array([0]), values=np.full(n * n, value))


@pytest.mark.parametrize("products", ["f64", "sliced_bf16"])
def test_infinite_ritz_value(products):
    X = torch.full((1, 2), 1e-10, dtype=torch.float64, device="cuda")
    with D.Context(one_element(2, 1e308)) as ctx:
        ctx.set_subspace_products(products)
        with pytest.raises(D.DGChefsiError) as e:
            ctx.cycle(X, 1, 1.0, 0.01, bounds=(0.0, 1.0, -1e298))
        assert e.value.status in ("ERR_NONFINITE", "ERR_NO_CONVERGENCE")
        assert bool((X == 1e-10).all())
        # the same cycle on a smaller H, with the same context
        ctx.set_values(torch.full((4,), 3.0, dtype=torch.float64, device="cuda"))
        out = ctx.cycle(X, 1, 1.0, 0.01, bounds=(0.0, 1.0, -2.0))
        assert abs(float(out["ritz"][0]) - 6.0) < 1e-12 and abs(float(X.norm()) - 1.0) < 1e-12


@pytest.mark.parametrize("products", ["f64", "sliced_bf16"])
def test_zero_state(products):
    """A state of zeros stays one through the filter: a pivot of exactly zero."""
    cfg = G.scaled_copy(G.CONFIGS["bulk3d_8x8x8"], grid=(2, 2, 2), nb=16, Ns=8)
    H = G.make_blocks(cfg)
    X0 = torch.from_numpy(np.random.default_rng(1).standard_normal((8, H.N))).cuda()
    X0[5] = 0.0
    X = X0.clone()
    with D.Context(H) as ctx:
        ctx.set_subspace_products(products)
        with pytest.raises(D.DGChefsiError) as e:
            ctx.cycle(X, 3, 4.0, 0.05, bounds=(5.0, 45.0, -1.7))
        assert e.value.status == "ERR_NOT_SPD" and torch.equal(X, X0)
