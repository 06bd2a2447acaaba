"""Warp-staged hops whose streams are evict-first in L2 (GPU vs oracle).

A timeslice of the hop's input just above and just below the 8 MB at which the policy
changes, at widths 32 and 16.  The FP32 hop is held to a few units of 2^-24 of the
largest output (48 products of rounded inputs); the solve to its tolerance by the
oracle's FP64 M.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims, n, kind", [((18, 18, 18, 2), 31, 11), ((18, 18, 16, 2), 31, 11), ((18, 18, 18, 2), 32, 4),
                                           ((22, 22, 24, 2), 15, 12)])
def test_streams(lib, dims, n, kind):
    kappa, N = 0.11, 1 << (n - 1).bit_length()
    U = synthetic.gauge_field(dims, eps=0.45, seed=99)
    b = synthetic.random_spinor(dims, seed=100, n=n)
    bt = torch.from_numpy(b).cuda()
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    assert c.tune_hop(1, N, force_pf=kind)[2] == kind
    h = c.apply_hop(bt, precision=1).cpu().numpy()
    x, st = c.solve(bt, lib.Params(tol=1e-11, precision=1, batch=N))
    assert all(s["status"] == 0 for s in st), st
    for j in (0, n - 1):
        ref = wilson.hop(U, b[j], -1.0)
        assert np.abs(h[j] - ref).max() < 1e-6 * np.abs(ref).max()
        r = b[j] - wilson.apply_m(U, x[j].cpu().numpy(), kappa, -1.0)
        assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b[j])
    c.close()
