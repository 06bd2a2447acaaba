"""Clover solves form their residuals in FP64: the switch for float-float steps does not reach them (GPU)."""

import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [1, 2])
def test_clover_defect_correction_is_fp64(lib, prec, monkeypatch):
    dims = (4, 4, 4, 6)
    c = lib.Context(dims)
    c.load_gauge(synthetic.gauge_field(dims, eps=0.45, seed=77))
    c.set_kappa(0.11)
    c.set_clover(1.2)
    b = torch.from_numpy(synthetic.random_spinor(dims, seed=78, n=5)).cuda()
    sols = []
    for flag in ("1", "0"):
        monkeypatch.setenv("DLOOPS_OUTER_DFF", flag)
        x, st = c.solve(b, lib.Params(tol=1e-10, precision=prec, batch=8))
        assert all(s["status"] == 0 for s in st), st
        sols.append(x)
    assert torch.equal(*sols)
    c.close()
