"""The FP64 hop with four warps to a site, on both sides of the sizes where it takes over (GPU vs oracle).

Widths 1 to 64 (one group of 32 items a block, two, and the whole-site kernel),
site counts that fill no whole group, fields of unequal right-hand sides.  Bound:
FP64 sums of 48 products, 1e-13 of the largest value.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims, n", [((2, 2, 2, 2), 1), ((2, 2, 2, 2), 64), ((6, 2, 4, 6), 3), ((6, 6, 6, 6), 8),
                                     ((8, 8, 8, 18), 1), ((8, 8, 8, 20), 2), ((4, 4, 4, 4), 64), ((4, 6, 4, 4), 64)])
def test_fp64_hop_and_solve(lib, dims, n):
    kappa = 0.11
    U = synthetic.gauge_field(dims, eps=0.45, seed=81)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    psi = synthetic.random_spinor(dims, seed=82, n=n)
    psi *= (1.0 + np.arange(n)).reshape(-1, 1, 1, 1, 1, 1, 1)
    x = torch.from_numpy(psi).cuda()
    ref = wilson.hop(U, psi, -1.0)
    assert np.abs(c.apply_hop(x).cpu().numpy() - ref).max() < 1e-13 * np.abs(ref).max()
    assert np.abs(c.apply_m(x).cpu().numpy() - (psi - kappa * ref)).max() < 1e-13 * np.abs(ref).max()
    for method in (0, 1):  # the fused reductions of both methods
        sol, st = c.solve(x, lib.Params(tol=1e-12, precision=0, batch=64, method=method))
        assert all(s["status"] == 0 for s in st), st
        sol = sol.cpu().numpy()
        for j in {0, n - 1}:
            r = psi[j] - wilson.apply_m(U, sol[j], kappa, -1.0)
            assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(psi[j])
    c.close()
