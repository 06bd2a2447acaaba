"""Width-16 hops with two sites per warp, and last batches in a narrower layout (GPU vs oracle).

8^3 x 24 has 3072 pairs of sites, more than the warps of a launch, so every warp
walks several; 2^3 x 4 has 8 pairs.  The FP32 hop is held to a few units of 2^-24
of the largest output (48 products of rounded inputs).
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (6, 2, 4, 6), (8, 8, 8, 24)])
def test_two_sites_per_warp(lib, dims):
    kappa = 0.11
    U = synthetic.gauge_field(dims, eps=0.45, seed=91)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    R, B, kind, _ = c.tune_hop(1, 16, force_pf=12)
    assert kind == 12 and all(c.hop_shape(1, 16, k)[2] == 12 for k in (0, 1, 2))
    with pytest.raises(lib.DlError):
        c.set_hop_shape(1, 16, 0, 1, 64, 12)
    b = synthetic.random_spinor(dims, seed=92, n=15)
    bt = torch.from_numpy(b).cuda()
    ref = wilson.hop(U, b, -1.0)
    assert np.abs(c.apply_hop(bt, precision=1).cpu().numpy() - ref).max() < 1e-6 * np.abs(ref).max()
    for method in (0, 1):
        x, st = c.solve(bt, lib.Params(tol=1e-11, precision=1, batch=16, method=method))
        assert all(s["status"] == 0 for s in st), st
        x = x.cpu().numpy()
        for j in (0, 14):
            r = b[j] - wilson.apply_m(U, x[j], kappa, -1.0)
            assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b[j])
    c.close()


@pytest.mark.parametrize("prec, n", [(1, 33), (1, 41), (2, 35)])
def test_narrow_last_batch(lib, prec, n):
    """A last batch of 1, 9 or 3 right-hand sides after a full one of 32 (12^3 x 16: solved step by step)."""
    dims, kappa = (12, 12, 12, 16), 0.11
    U = synthetic.gauge_field(dims, eps=0.45, seed=93)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    b = c.make_sources(seed=8, noise_first=0, n_noise=n, dilution=0)
    x, st = c.solve(b, lib.Params(tol=1e-11, precision=prec, batch=32))
    assert all(s["status"] == 0 for s in st), st
    r = b - c.apply_m(x)
    assert (r.flatten(1).norm(dim=1) <= 1.01e-11 * b.flatten(1).norm(dim=1)).all()
    j = n - 1
    xj = x[j].cpu().numpy()[None]
    rj = b[j].cpu().numpy()[None] - wilson.apply_m(U, xj, kappa, -1.0)
    assert np.linalg.norm(rj) <= 1e-11 * np.linalg.norm(b[j].cpu().numpy())
    y, _ = c.solve_adjoint(b[32:].contiguous(), lib.Params(tol=1e-11, precision=prec, batch=32))
    rj = b[j].cpu().numpy()[None] - wilson.apply_mdag(U, y[-1].cpu().numpy()[None], kappa, -1.0)
    assert np.linalg.norm(rj) <= 1e-11 * np.linalg.norm(b[j].cpu().numpy())
    c.close()
