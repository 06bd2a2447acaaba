"""One-launch solves with clusters of 1 to 16 blocks, each at the fewest sites that size takes (GPU vs oracle).

A cluster of C blocks starts at 128 (C / 2) + 8 even sites, where the blocks hold the fewest sites and reach
their first exchange through each other's shared memory soonest after the launch.  Many short solves, each
of them a launch per cycle, have to meet their tolerance by the oracle's FP64 M and to be equal bit by bit.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 34), (2, 2, 2, 66), (2, 2, 2, 130), (2, 2, 4, 130)])
@pytest.mark.parametrize("prec, method", [(1, 0), (2, 0), (1, 1)])
def test_smallest_clusters(lib, dims, prec, method):
    kappa, tol = 0.11, 1e-10
    U = synthetic.gauge_field(dims, eps=0.45, seed=55)
    b = synthetic.random_spinor(dims, seed=56, n=2)
    bt = torch.from_numpy(b).cuda()
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(kappa)
    p = lib.Params(tol=tol, precision=prec, batch=2, method=method)
    x, st = c.solve(bt, p)
    assert all(s["status"] == 0 for s in st), st
    for _ in range(50):
        assert torch.equal(c.solve(bt, p)[0], x)
    x = x.cpu().numpy()
    for j in range(2):
        r = b[j] - wilson.apply_m(U, x[j], kappa, -1.0)
        assert np.linalg.norm(r) <= tol * np.linalg.norm(b[j])
    c.close()
