"""The 64-row leaf and the 8 x 8 small products of the recursive Cholesky at
their edges: orders around the 8-row tile and the 64-row leaf, padded rows of
the matrix, a non-positive pivot in every tile position."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def tiny_ctx():
    ctx = D.Context(G.make_blocks(G.CONFIGS["tiny_2x2x2"]))
    ctx.set_cholesky("products")
    return ctx


def strided(S, pad):
    n = S.shape[0]
    big = torch.full((n, n + pad), float("nan"), dtype=torch.float64, device="cuda")
    big[:, :n] = torch.from_numpy(np.tril(S) + np.triu(np.full((n, n), np.nan), 1)).cuda()  # upper part not read
    return big[:, :n]


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 31, 56, 57, 63, 64, 65, 72, 100, 127, 128, 129, 191, 200])
def test_inverse_factor_at_tile_edges(n):
    """L^{-1} against the exact factor's inverse in FP64: both are within
    n u cond of the truth; 1e3 is the planted condition number."""
    S, _ = G.planted_cholesky(n, 1e3, seed=n)
    ref = np.linalg.inv(np.linalg.cholesky(S))
    with tiny_ctx() as ctx:
        got = np.tril(ctx.cholesky_inverse(strided(S, 5)).cpu().numpy())
    assert np.max(np.abs(got - ref)) <= 8 * n * 2.0 ** -53 * 1e3 * np.max(np.abs(ref))


@pytest.mark.parametrize("n,col", [(1, 0), (8, 7), (20, 0), (64, 1), (64, 8), (64, 31), (64, 63), (70, 64), (70, 69),
                                   (129, 100), (129, 128)])
def test_bad_pivot_reports_its_column(n, col):
    S, _ = G.planted_cholesky(n, 1e2, negative_at=col, seed=col)
    with tiny_ctx() as ctx:
        with pytest.raises(D.DGChefsiError) as e:
            ctx.cholesky_inverse(strided(S, 0))
    assert e.value.status == "ERR_NOT_SPD" and f"column {col + 1} " in str(e.value) + " "


def test_extreme_scales():
    """Diagonals over 200 orders of magnitude: equilibrated exactly, and the
    pivots' reciprocal roots stay in range."""
    n = 90
    S, _ = G.planted_cholesky(n, 1e2, seed=1)
    d = 2.0 ** np.linspace(-330, 330, n).round()
    with tiny_ctx() as ctx:
        a = np.tril(ctx.cholesky_inverse(strided(S, 0)).cpu().numpy())
        b = np.tril(ctx.cholesky_inverse(strided(S * d[:, None] * d[None, :], 0)).cpu().numpy())
    # (D L)^{-1} = L^{-1} D^{-1}, and powers of two change no rounding
    assert np.allclose(b * d[None, :], a, rtol=1e-12, atol=1e-14)
