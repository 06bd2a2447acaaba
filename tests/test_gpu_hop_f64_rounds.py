"""The FP64 hop of whole sites with few and with many blocks per SM (GPU vs oracle).

On 152 SMs: 6.7, 8.4 and 10.1 blocks of 64 (site, right-hand side) items an SM, which take the kernels for six
resident blocks, for five, and for five at the end of that range.  Bound: FP64 sums of 48 products, 1e-13 of
the largest value; the solves to their tolerance by the oracle's M.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims, n", [((8, 8, 8, 16), 15), ((8, 8, 8, 20), 15), ((8, 8, 8, 24), 16)])
def test_fp64_hop_rounds(lib, dims, n):
    kappa = 0.11
    U = synthetic.gauge_field(dims, eps=0.45, seed=83)
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    psi = synthetic.random_spinor(dims, seed=84, n=n)
    x = torch.from_numpy(psi).cuda()
    h = c.apply_hop(x).cpu().numpy()
    m = c.apply_m(x).cpu().numpy()
    for j in (0, n - 1):
        ref = wilson.hop(U, psi[j], -1.0)
        assert np.abs(h[j] - ref).max() < 1e-13 * np.abs(ref).max()
        assert np.abs(m[j] - (psi[j] - kappa * ref)).max() < 1e-13 * np.abs(ref).max()
    for method in (0, 1):
        sol, st = c.solve(x, lib.Params(tol=1e-12, precision=0, batch=16, method=method))
        assert all(s["status"] == 0 for s in st), st
        r = psi[n - 1] - wilson.apply_m(U, sol[n - 1].cpu().numpy(), kappa, -1.0)
        assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(psi[n - 1])
    c.close()
