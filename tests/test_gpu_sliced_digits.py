"""The 9-bit digits of the dense sliced products: bit for bit at the edge of the
exact FP32 sums, at ragged drains of the accumulator (256 terms, or more where
the digits' norms allow), at ragged K chunks and tiles, on operands whose
digits are all in use, and the one rounding of the digit sums."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def product(A, Bt, b_rows, slices=10):
    with D.Context(G.make_blocks(G.CONFIGS["tiny_2x2x2"])) as ctx:
        B = Bt if b_rows else np.ascontiguousarray(Bt.T)
        out = ctx.sliced_gemm(torch.from_numpy(A.astype(np.float64)).cuda(), torch.from_numpy(B.astype(np.float64)).cuda(),
                              b_rows=b_rows, slices=slices)
        return out.cpu().numpy()


@pytest.mark.parametrize("b_rows", [True, False])
@pytest.mark.parametrize("M,Nc,K", [(1, 1, 255), (3, 130, 256), (257, 5, 257), (70, 301, 512), (255, 257, 1030),
                                    (40, 50, 4096), (33, 20, 4097), (129, 64, 8500)])
def test_digits_at_their_bounds_bit_exact(M, Nc, K, b_rows):
    """130816 = 2^17 - 256 splits (exponent 17) into q_0 = 256, q_1 = -256, so
    products of equal-sign rows sum to +-256^3 = +-2^24 over 256 terms; rows of
    mixed sign and a row of ones beside them. The exact products are integers
    below 2^53."""
    rng = np.random.default_rng(1)
    A = np.full((M, K), 130816, dtype=np.int64)
    Bt = np.full((Nc, K), 130816, dtype=np.int64)
    A[1::3] *= -1
    Bt[1::4] *= rng.choice([-1, 1], size=K)
    if M > 2:
        A[2] = 1
    assert np.array_equal(product(A, Bt, b_rows), (A @ Bt.T).astype(np.float64))


@pytest.mark.parametrize("slices", [4, 7, 10, 12])
@pytest.mark.parametrize("M,Nc,K", [(300, 131, 4096), (64, 700, 1000), (513, 259, 5000)])
def test_random_integers_bit_exact(M, Nc, K, slices):
    """Random integers of 6 a and 6 b bits, a + b <= slices + 1, that `slices`
    slices multiply exactly (the product stays below 2^53)."""
    rng = np.random.default_rng(2)
    a = min(slices // 2, 3)
    b = min(slices + 1 - a, 3)
    A = rng.integers(-(2 ** (6 * a - 1)), 2 ** (6 * a - 1), size=(M, K))
    Bt = rng.integers(-(2 ** (6 * b - 1)), 2 ** (6 * b - 1), size=(Nc, K))
    assert np.array_equal(product(A, Bt, True, slices), (A @ Bt.T).astype(np.float64))


@pytest.mark.parametrize("slices", [10, 11])
@pytest.mark.parametrize("M,Nc,K,e", [(1, 1, 700, 0), (5, 7, 700, -537), (40, 301, 300, 400), (257, 64, 513, -40)])
def test_sums_are_rounded_once(M, Nc, K, e, slices):
    """Integers of 27 bits have four digits at most and no pair of them is
    dropped, so the sum (up to 64 bits) is exact before its only rounding:
    the result is the nearest double, ties to even. e scales both operands by
    2^e; at -537 small integers end as exact subnormals. One K chunk."""
    rng = np.random.default_rng(3)
    top = 2 ** 27 if e != -537 else 2 ** 8
    A = rng.integers(-top, top, size=(M, K))
    Bt = rng.integers(-top, top, size=(Nc, K))
    if M > 1:
        A[1] = 0
        Bt[::3] = abs(Bt[::3])
        A[0] = abs(A[0])
    exact = A.astype(object) @ Bt.T.astype(object)
    want = np.array([[float(x) for x in row] for row in exact])
    assert np.array_equal(product(A * 2.0 ** e, Bt * 2.0 ** e, True, slices), np.ldexp(want, 2 * e))


@pytest.mark.parametrize("grid,nb,Ns,ld_more", [((1, 1, 1), 5, 1, 0), ((3, 2, 2), (17, 31), 9, 1), ((4, 2, 2), 64, 5, 0),
                                                ((3, 3, 2), 70, 4, 3), ((5, 7, 1), (40, 120), 3, 1)])
def test_state_digits_bit_exact(grid, nb, Ns, ld_more):
    """Integer H and states (products far below 2^53) on states of 1 to 58
    slices of 64, slices that are not full, rows and elements that start on 8 or 16
    bytes: the sliced H X equals the FP64 product bit for bit."""
    cfg = G.scaled_copy(G.CONFIGS["sheet2d_24x20" if grid[2] == 1 else "bulk3d_8x8x8"], grid=grid, nb=nb, Ns=Ns)
    H = G.make_blocks(cfg)
    rng = np.random.default_rng(5)
    X = torch.zeros((Ns, H.N + ld_more), dtype=torch.float64, device="cuda")
    X[:, : H.N] = torch.from_numpy(rng.integers(-2 ** 20, 2 ** 20, size=(Ns, H.N)).astype(np.float64)).cuda()
    with D.Context(H) as ctx:
        ctx.set_values(torch.from_numpy(np.round(H.values * 64)).cuda())
        W, V = torch.zeros_like(X), torch.zeros_like(X)
        ctx.sliced_matvec(X[:, : H.N], W[:, : H.N])
        ctx.matvec(X[:, : H.N], V[:, : H.N])
        assert torch.equal(W, V)
