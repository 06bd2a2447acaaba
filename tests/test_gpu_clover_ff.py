"""Float-float defect correction of the clover operator (GPU vs oracle).

Widths and site counts at the edges (one right-hand side, a ragged batch, 64), sources
from 1e-42 to 1e35 in one batch, both inner precisions, float-float and FP64 steps
(DLOOPS_OUTER_DFF=0): each solution meets tol by the oracle's FP64 M, and the two
agree within 2 tol cond(M) (cond(M) < 20 at kappa 0.11).
"""

import numpy as np
import pytest

import synthetic
from oracle import clover

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims, n, batch", [((2, 2, 2, 4), 1, 1), ((4, 2, 6, 4), 5, 8), ((4, 4, 4, 4), 33, 64)])
@pytest.mark.parametrize("prec", [1, 2])
def test_clover_float_float_steps(lib, dims, n, batch, prec, monkeypatch):
    kappa, csw, tol = 0.11, 1.2, 1e-10
    U = synthetic.gauge_field(dims, eps=0.45, seed=95)
    b = synthetic.random_spinor(dims, seed=96, n=n)
    scale = np.array([1e-42, 1.0, 1e35, 1e-7] * 17)[:n]
    b *= scale.reshape(-1, 1, 1, 1, 1, 1, 1)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    c.set_clover(csw)
    sols = []
    for flag in ("1", "0"):
        monkeypatch.setenv("DLOOPS_OUTER_DFF", flag)
        x, st = c.solve(torch.from_numpy(b).cuda(), lib.Params(tol=tol, precision=prec, batch=batch))
        assert all(s["status"] == 0 for s in st), st
        x = x.cpu().numpy()
        for j in {0, n // 2, n - 1}:
            r = b[j] - clover.apply_m(U, x[j], kappa, csw)
            assert np.linalg.norm(r / scale[j]) <= tol * np.linalg.norm(b[j] / scale[j])
        sols.append(x / scale.reshape(-1, 1, 1, 1, 1, 1, 1))
    assert np.linalg.norm(sols[0] - sols[1]) <= 40 * tol * np.linalg.norm(sols[1])
    c.set_kappa(0.1)  # the blocks are rebuilt in both formats
    monkeypatch.setenv("DLOOPS_OUTER_DFF", "1")
    x, st = c.solve(torch.from_numpy(b).cuda(), lib.Params(tol=tol, precision=prec, batch=batch))
    r = b[-1] - clover.apply_m(U, x[-1].cpu().numpy(), 0.1, csw)
    assert np.linalg.norm(r / scale[-1]) <= tol * np.linalg.norm(b[-1] / scale[-1])
    c.close()
