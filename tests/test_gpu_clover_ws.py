"""Warp-staged clover hops at widths 32 and 16 (GPU vs the FP64 direct kernel and the oracle).

16 to 6144 sites per parity: fewer sites than the warps of a launch, and several per
warp.  Four BiCGStab iterations in FP32 and in FP64 take the same steps; their
rounding errors (2^-24 per operation, amplified by at most cond(M)^2 < 400 a step,
a few hundred operations each) stay below 1e-3, a misplaced element does not.
"""

import numpy as np
import pytest

import synthetic
from oracle import clover

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (6, 2, 4, 6), (8, 8, 8, 24)])
@pytest.mark.parametrize("n, batch", [(29, 32), (13, 16)])
def test_clover_warp_staged(lib, dims, n, batch):
    kappa, csw = 0.11, 1.2
    U = synthetic.gauge_field(dims, eps=0.45, seed=97)
    b = synthetic.random_spinor(dims, seed=98, n=n)
    bt = torch.from_numpy(b).cuda()
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    c.set_clover(csw)
    xs = [c.solve(bt, lib.Params(precision=p, fixed_iters=4, batch=batch))[0] for p in (0, 1)]
    assert ((xs[1] - xs[0]).flatten(1).norm(dim=1) <= 1e-3 * xs[0].flatten(1).norm(dim=1)).all()
    x, st = c.solve(bt, lib.Params(tol=1e-11, precision=1, batch=batch))
    assert all(s["status"] == 0 for s in st), st
    for j in (0, n - 1):
        r = b[j] - clover.apply_m(U, x[j].cpu().numpy(), kappa, csw)
        assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b[j])
    c.close()
