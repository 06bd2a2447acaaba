"""Warp-staged hops at width 64 and with the clover term on both sides of the evict-first line (GPU vs oracle).

A timeslice of the input above and below 8 MB; every kernel that the stage counts, the width and the streams
select.  The FP32 hop is held to a few units of 2^-24 of the largest output (48 products of rounded inputs),
the solves of both methods to their tolerance by the oracle's FP64 M.
"""

import numpy as np
import pytest

import synthetic
from oracle import clover, wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(14, 14, 14, 2), (14, 14, 12, 2)])
@pytest.mark.parametrize("kind", [4, 11])
def test_width_64(lib, dims, kind):
    kappa, n = 0.11, 61
    U = synthetic.gauge_field(dims, eps=0.45, seed=101)
    b = synthetic.random_spinor(dims, seed=102, n=n)
    bt = torch.from_numpy(b).cuda()
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    for k in range(3):
        c.set_hop_shape(1, n, k, 2, 64, kind)
    h = c.apply_hop(bt, precision=1).cpu().numpy()
    for j in (0, n - 1):
        ref = wilson.hop(U, b[j], -1.0)
        assert np.abs(h[j] - ref).max() < 1e-6 * np.abs(ref).max()
    for method in (0, 1):
        x, st = c.solve(bt, lib.Params(tol=1e-11, precision=1, batch=64, method=method))
        assert all(s["status"] == 0 for s in st), st
        for j in (0, n - 1):
            r = b[j] - wilson.apply_m(U, x[j].cpu().numpy(), kappa, -1.0)
            assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b[j])
    c.close()


@pytest.mark.parametrize("dims, n", [((18, 18, 18, 2), 31), ((18, 18, 16, 2), 31), ((22, 22, 24, 2), 15), ((22, 22, 16, 2), 15)])
def test_clover(lib, dims, n):
    kappa, csw = 0.11, 1.1
    U = synthetic.gauge_field(dims, eps=0.45, seed=103)
    b = synthetic.random_spinor(dims, seed=104, n=n)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    c.set_clover(csw)
    x, st = c.solve(torch.from_numpy(b).cuda(), lib.Params(tol=1e-10, precision=1, batch=32))
    assert all(s["status"] == 0 for s in st), st
    for j in (0, n - 1):
        r = b[j] - clover.apply_m(U, x[j].cpu().numpy(), kappa, csw)
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b[j])
    c.close()
