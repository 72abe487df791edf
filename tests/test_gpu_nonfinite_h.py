"""Values of H that are not finite (set_values does not check them): every sliced
call reports them, not only the first one after them, and the next finite values
give the bits of a new context."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("slices", [10, 12])
def test_reported_by_every_call(bad, slices):
    cfg = G.scaled_copy(G.CONFIGS["bulk3d_8x8x8"], grid=(3, 2, 2), nb=(17, 40), Ns=30)
    H = G.make_blocks(cfg)
    X = torch.from_numpy(np.random.default_rng(1).standard_normal((30, H.N))).cuda()
    good = torch.from_numpy(H.values).cuda()
    broken = good.clone()
    broken[int(H.blk_off[5]) + 3] = bad
    with D.Context(H) as ctx, D.Context(H) as new:
        ctx.set_subspace_products("sliced_bf16", slices)
        ctx.sliced_matvec(X, slices=slices)
        ctx.set_values(broken)
        for call in (lambda: ctx.sliced_matvec(X, slices=slices), lambda: ctx.rayleigh_ritz(X.clone())):
            for _ in range(2):
                with pytest.raises(D.DGChefsiError) as e:
                    call()
                assert e.value.status == "ERR_NONFINITE"
        # nor does a state that is not finite spoil the digits of H formed beside it
        ctx.set_values(good)
        Xbad = X.clone()
        Xbad[3, 4] = bad
        with pytest.raises(D.DGChefsiError):
            ctx.sliced_matvec(Xbad, slices=slices)
        assert torch.equal(ctx.sliced_matvec(X, slices=slices), new.sliced_matvec(X, slices=slices))
