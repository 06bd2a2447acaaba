"""Every launch shape that hop_shape reports is one that set_hop_shape takes (GPU)."""

import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (4, 4, 4, 8)


@pytest.fixture
def ctx(lib):
    c = lib.Context(DIMS)
    c.load_gauge(synthetic.gauge_field(DIMS, eps=0.45, seed=59))
    c.set_kappa(0.11)
    yield c
    c.close()


def set_again(c, prec, n):
    for cls in (0, 1, 2):
        shape = c.hop_shape(prec, n, cls)
        c.set_hop_shape(prec, n, cls, *shape)
        assert c.hop_shape(prec, n, cls) == shape


@pytest.mark.parametrize("prec, n", [(0, 1), (0, 64), (1, 1), (1, 16), (1, 32), (1, 64), (2, 1), (2, 16), (2, 32)])
@pytest.mark.parametrize("kind", range(-1, 13))
def test_tuned_shapes(lib, ctx, prec, n, kind):
    try:
        ctx.tune_hop(prec, n, force_pf=kind)
    except lib.DlError:
        pytest.skip("kind not built for this storage layout")
    set_again(ctx, prec, n)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_untuned_shapes(ctx, prec):
    for n in (1, 2, 4, 8, 16, 32, 64):
        set_again(ctx, prec, n)


@pytest.mark.parametrize("prec, n", [(0, 1), (0, 3), (1, 1), (1, 16), (2, 2)])
def test_shapes_after_a_solve(lib, ctx, prec, n):
    """Also where the solve tunes nothing: FP64, and small lattices in one launch per cycle."""
    b = torch.from_numpy(synthetic.random_spinor(DIMS, seed=60, n=n)).cuda()
    p = lib.Params(tol=1e-10, precision=prec, batch=n)
    x, _ = ctx.solve(b, p)
    set_again(ctx, prec, n)
    y, st = ctx.solve(b, p)
    assert all(s["status"] == 0 for s in st) and (x - y).norm() <= 1e-8 * x.norm()
