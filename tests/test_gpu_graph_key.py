"""Captured iterations of one context are told apart by precision and by method (GPU vs oracle)."""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order", [((1, 0), (0, 1)), ((0, 1), (1, 0))])
def test_paired_fp32_bicgstab_and_fp64_cgnr_in_one_context(lib, order, monkeypatch):
    """FP32 fields in the paired layout under BiCGStab, and FP64 ones under CGNR, at one width and chunk."""
    monkeypatch.setenv("DLOOPS_F32_PAIRS", "1")
    dims, kappa, tol = (4, 4, 4, 6), 0.11, 1e-10
    U = synthetic.gauge_field(dims, eps=0.45, seed=57)
    b = synthetic.random_spinor(dims, seed=58, n=4)
    bt = torch.from_numpy(b).cuda()
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    for prec, method in order:
        x, st = c.solve(bt, lib.Params(tol=tol, precision=prec, method=method, batch=4, chunk=2, use_graph=1))
        assert all(s["status"] == 0 for s in st), st
        x = x.cpu().numpy()
        for j in range(4):
            r = b[j] - wilson.apply_m(U, x[j], kappa, -1.0)
            assert np.linalg.norm(r) <= tol * np.linalg.norm(b[j])
    c.close()
