"""The reciprocal root of the Cholesky leaf's pivots against 1 / sqrt(p) in more
precision: mantissas over [1/4, 4) with both parities of the exponent and their
ends, and pivots on both sides of 2^-100, where the library's root takes over.

Tolerance: y = the FP32 root has a relative error below 2^-21, e = 1 - p y^2 is
off by at most 2^-53 (p y is rounded once, the rest is fused), which the step
halves; the series leaves 5/16 e^3 < 2^-61 and the last fused step rounds once:
1.5 x 2^-53 and a little. Powers of two are exact on both sides. The library's
root is documented to 1 unit in the last place. 2 x 2^-53 covers either."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu
TOL = 2.0 ** -52


def inverse_factor(S):
    with D.Context(G.make_blocks(G.CONFIGS["tiny_2x2x2"])) as ctx:
        ctx.set_cholesky("products")
        return np.tril(ctx.cholesky_inverse(torch.from_numpy(S).cuda()).cpu().numpy())


def relative_error(y, p):
    """|y sqrt(p) - 1| from the exact integers y^2 p."""
    out = []
    for a, b in zip(y, p):
        ma, ea = np.frexp(a)
        mb, eb = np.frexp(b)
        n = int(ma * 2 ** 53) ** 2 * int(mb * 2 ** 53)
        k = 3 * 53 - 2 * int(ea) - int(eb)  # y^2 p = n 2^-k, close to 1
        out.append(abs((n - (1 << k)) / (1 << k)) / 2)
    return np.array(out)


def test_mantissas():
    u = 2.0 ** -52
    ends = [m * s for s in (0.25, 0.5, 1.0, 2.0) for m in (1.0, 1.0 + u, 1.5 - u, 1.5, 2.0 - u, 2.0 - 2 * u)]
    # one below and above the values whose leading 23 bits are cut off next
    cut = [1.0 + k * 2.0 ** -23 + d * u for k in (1, 3, 2 ** 22 - 1, 2 ** 23 - 1) for d in (-1, 0, 1)]
    p = np.concatenate([ends, cut, np.random.default_rng(1).uniform(0.25, 4.0, 4000)])
    p = p[:len(p) // 8 * 8]
    worst = 0.0
    for part in np.array_split(p, 8):
        got = inverse_factor(np.diag(part))
        assert np.count_nonzero(got - np.diag(np.diag(got))) == 0
        worst = max(worst, relative_error(np.diag(got), part).max())
    assert worst <= TOL, worst


@pytest.mark.parametrize("residual", [7, 15, 23, 31, 39])
def test_tiny_pivots(residual):
    """l = A 2^-52 with A^2 = -residual modulo 2^53: S = [[1, l], [l, l^2 + residual
    2^-104]] has exact entries and the second pivot residual x 2^-104, which is
    below 2^-100 for 7 and 15 (the library's root) and above it for the others."""
    A = 1
    for k in range(3, 54):  # A^2 + residual = 0 modulo 2^k (residual = 7 modulo 8)
        if (A * A + residual) % (1 << k):
            A += 1 << (k - 2)
    A = next(a for a in ((A % 2 ** 52) + 2 ** 52, (-A % 2 ** 52) + 2 ** 52) if a * a < 2 ** 105)  # -A and + 2^52 solve it too
    a22 = A * A + residual  # times 2^-104: in [1, 2), so the equilibration scales nothing
    assert a22 % 2 ** 53 == 0
    S = np.array([[1.0, np.ldexp(float(A), -52)], [np.ldexp(float(A), -52), np.ldexp(float(a22), -104)]])
    assert int(np.ldexp(S[1, 1], 52)) << 52 == a22 and int(np.ldexp(S[0, 1], 52)) == A
    got = inverse_factor(S)
    assert got[0, 0] == 1.0
    assert relative_error([got[1, 1]], [np.ldexp(float(residual), -104)])[0] <= TOL
    assert abs(got[1, 0] / (-S[1, 0] * got[1, 1]) - 1.0) <= 2 * TOL
