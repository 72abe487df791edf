"""Which form the density blocks of a sliced cycle take. The FP64 form has the bits
of density_blocks; the digits' form has others (a sum of some hundred terms rounded
once against one rounding a term). Relative to sqrt(P_jj P_j'j') >= sum_i f_i |x_ij
x_ij'|, u = 2^-53: the FP64 sum is off by (Ns + 1) u; the digits' by two roundings
in each factor and one a chunk, 5 u, and by their remainders and the dropped pairs,
4 Ns (d + 2) 2^-9d, less than Ns u / 20 from d = 7 on. 2 (Ns + 8) u covers both."""
import numpy as np
import pytest
import torch

import fake_cuda_malloc
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def cycle(grid, nb, Ns, slices, kT=0.05):
    """(P of the cycle, density_blocks of its states and occupations, their difference over sqrt(P_jj P_j'j'))."""
    cfg = G.scaled_copy(G.CONFIGS["bulk3d_8x8x8" if grid[2] > 1 else "sheet2d_24x20"], grid=grid, nb=nb, Ns=Ns)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(4)
    with D.Context(H) as ctx:
        ctx.set_subspace_products("sliced_bf16", slices)
        X = torch.from_numpy(rng.standard_normal((Ns, H.N))).cuda()
        out = ctx.cycle(X, m=4, Ne=1.1 * Ns, kT=kT, v0=torch.from_numpy(rng.standard_normal(H.N)).cuda(), prec="f64")
        Q = ctx.density_blocks(X, out["f"])
        worst = 0.0
        for p, q in zip(ctx.unpack_density(out["P"]), ctx.unpack_density(Q)):
            d = q.diagonal().sqrt()
            worst = max(worst, float(((p - q).abs() / (d[:, None] * d[None, :])).max()))
    return out["P"], Q, worst


@pytest.mark.parametrize("slices", [10, 11, 12, 13, 14, 16])
def test_digits_of_every_count(slices):
    """7 to 11 digits, on either side of the 64-bit splitting (7)."""
    P, Q, worst = cycle((4, 4, 3), (30, 60), 1100, slices)
    assert not torch.equal(P, Q)
    assert worst <= 2 * (1100 + 8) * 2.0 ** -53


@pytest.mark.parametrize("grid,nb,Ns,digits", [((4, 4, 4), 40, 500, False), ((4, 4, 4), 64, 600, True),
                                               ((6, 6, 6), 8, 1300, False), ((6, 6, 6), 16, 900, False),
                                               ((6, 6, 6), 17, 900, True)])
def test_rule(grid, nb, Ns, digits):
    """Enough states, and 16 functions an element and more on average over the packed
    rows: the last tile of 216 elements of 16 is half full, which puts them below."""
    P, Q, worst = cycle(grid, nb, Ns, 10)
    assert torch.equal(P, Q) != digits
    assert worst <= 2 * (Ns + 8) * 2.0 ** -53


@pytest.mark.parametrize("kT", [0.004, 1.0])
def test_uneven_occupations(kT):
    """Rows whose entries sqrt(f_i) x_ij fall off over many orders, to zero and slowly."""
    P, Q, worst = cycle((4, 4, 3), 64, 1100, 10, kT=kT)
    assert not torch.equal(P, Q) and worst <= 2 * (1100 + 8) * 2.0 ** -53


def test_without_memory_for_the_packed_rows(tmp_path):
    """Elements of 129 functions fill a 256-row tile each, so the packed rows (12 x
    256 x 1500 doubles) are larger than what the rotation allocated before them;
    refused, the FP64 form takes over."""
    out = fake_cuda_malloc.run(tmp_path, r"""
cfg = G.scaled_copy(G.CONFIGS["sheet2d_24x20"], grid=(4, 3, 1), nb=129, Ns=1500)
H = G.make_blocks(cfg)
rng = np.random.default_rng(4)
X = torch.from_numpy(rng.standard_normal((1500, H.N))).cuda()
v = torch.from_numpy(rng.standard_normal(H.N)).cuda()
size = 12 * 256 * 1500 * 8
for deny_it in (False, True):
    with D.Context(H) as ctx:
        ctx.set_subspace_products("sliced_bf16", 10)
        if deny_it:
            deny(size, size)
        Y = X.clone()
        out = ctx.cycle(Y, m=4, Ne=1650.0, kT=0.05, v0=v, prec="f64")
        print("form", torch.equal(out["P"], ctx.density_blocks(Y, out["f"])))
        deny(1, 0)
        Y = X.clone()  # and the same context goes on
        again = ctx.cycle(Y, m=4, Ne=1650.0, kT=0.05, v0=v, prec="f64")
        print("form", torch.equal(again["P"], ctx.density_blocks(Y, again["f"])))
""")
    assert [w for w in out.split() if w in ("True", "False")] == ["False", "False", "True", "False"]
