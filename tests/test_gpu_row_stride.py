"""Blocks whose rows are further apart than N, through the calls of the Python
binding whose output has the input's row stride: the output is allocated with it,
a given one must have it, and the values are those of a contiguous block."""
import numpy as np
import pytest
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G

pytestmark = pytest.mark.gpu


def blocks(Ns=9, pad=5):
    cfg = G.ProblemConfig(name="stride", grid=(3, 2, 2), periodic=(True, True, True), stencil="27", nb=(5, 12), Ns=Ns,
                          m=4, Ne=1.0, seed=3)
    H = G.make_blocks(cfg)
    X = torch.from_numpy(np.random.default_rng(1).standard_normal((Ns, H.N))).cuda()
    wide = torch.full((Ns, H.N + pad), 7.0, dtype=torch.float64, device="cuda")
    wide[:, :H.N] = X
    return H, X, wide, wide[:, :H.N]


@pytest.mark.parametrize("m", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("prec", ["f64", "bf16x3"])
def test_gradient(prec, m):
    H, X, wide, Xs = blocks()
    with D.Context(H) as ctx:
        E, ritz, Hb, Xb = ctx.energy_grad(X, m, 5.0, 46.0, -1.8, 9.0, 0.3, prec=prec)
        Es, ritzs, Hbs, Xbs = ctx.energy_grad(Xs, m, 5.0, 46.0, -1.8, 9.0, 0.3, prec=prec)
        assert ctx.energy_grad(Xs, m, 5.0, 46.0, -1.8, 9.0, 0.3, grad=False, prec=prec)[0] == E
    assert Xbs.stride() == Xs.stride() and Xbs.shape == X.shape
    assert Es == E and torch.equal(ritzs, ritz) and torch.equal(Hbs, Hb) and torch.equal(Xbs, Xb)
    assert bool((wide[:, H.N:] == 7.0).all())


@pytest.mark.parametrize("prec", ["f64", "tf32", "bf16x3"])
def test_graph_filter(prec):
    H, X, wide, Xs = blocks()
    with D.Context(H) as ctx:
        Y = ctx.filter(X, 4, 5.0, 46.0, -1.8, prec=prec)
        Ys = ctx.filter_graph(Xs, 4, 5.0, 46.0, -1.8, prec=prec)
        assert Ys.stride() == Xs.stride() and torch.equal(Ys, Y)
        with pytest.raises(ValueError):
            ctx.filter_graph(Xs, 4, 5.0, 46.0, -1.8, prec=prec, Y=torch.empty_like(X))
        with pytest.raises(ValueError):
            ctx.filter_graph(X, 4, 5.0, 46.0, -1.8, prec=prec, Y=wide[:, :H.N])
        with pytest.raises(ValueError):
            ctx.filter_graph(X, 4, 5.0, 46.0, -1.8, prec=prec, Y=torch.empty_like(X)[:-1])


def test_overlapping_rows_are_refused():
    """An expanded row has stride 0: it was read as a block of rows N apart."""
    H, X, wide, Xs = blocks()
    with D.Context(H) as ctx:
        for bad in (X[:1].expand(4, H.N), X.reshape(-1).as_strided((4, H.N), (H.N - 1, 1))):
            for call in (ctx.gram, ctx.matvec, lambda x: ctx.energy_grad(x, 2, 5.0, 46.0, -1.8, 2.0, 0.3)):
                with pytest.raises(ValueError):
                    call(bad)
            with pytest.raises(ValueError):
                ctx.filter_host(bad.cpu()[:1].expand(4, H.N), 2, 5.0, 46.0, -1.8)
        assert ctx.gram(X[:1].expand(1, H.N)).shape == (1, 1)
