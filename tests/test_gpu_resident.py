"""The cluster-resident solver against the oracle's M and against the step-by-step solver (GPU).

Small lattices run their inner phases in one launch, one thread-block cluster per
right-hand side.  The sizes here sit at its edges: fewer sites than a tile of 32,
sites that fill no whole tile, one block per cluster, clusters of 16, several
rounds of sites per block, more right-hand sides than lie in one batch.  Each
solve must meet its tolerance by the oracle's FP64 M; two solutions of relative
residual tol differ by at most 2 tol cond(M), and cond(M) <= (1 + 8 k)/(1 - 8 k)
in the free field (k = 0.11: 16), so 1e-9 bounds the difference at tol 1e-11.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims, n, batch", [((2, 2, 2, 2), 3, 4), ((4, 4, 4, 4), 64, 64), ((6, 2, 4, 6), 1, 1),
                                            ((6, 6, 6, 8), 5, 32), ((6, 10, 4, 12), 7, 4), ((8, 8, 8, 16), 1, 1),
                                            ((4, 6, 2, 4), 35, 32), ((256, 2, 2, 2), 2, 2),
                                            ((2, 256, 2, 4), 1, 1)])
@pytest.mark.parametrize("prec, method", [(1, 0), (2, 0), (1, 1)])
def test_resident_solve(lib, dims, n, batch, prec, method):
    kappa, tol = 0.11, 1e-11
    U = synthetic.gauge_field(dims, eps=0.45, seed=51)
    b = synthetic.random_spinor(dims, seed=52, n=n)
    b[0] = 0.0
    b[0].reshape(-1)[5] = 1.0  # a point source among the others
    bt = torch.from_numpy(b).cuda()
    sols = []
    for pinned in (False, True):
        c = lib.Context(dims)
        c.load_gauge(U)
        c.set_kappa(kappa)
        if pinned:  # a pinned launch shape keeps the solve step by step
            c.tune_hop(prec, batch, force_pf=0)
        p = lib.Params(tol=tol, precision=prec, batch=batch, method=method)
        x, st = c.solve(bt, p)
        again, _ = c.solve(bt, p)
        assert torch.equal(x, again)
        assert all(s["status"] == 0 and s["true_residual"] <= tol for s in st), st
        sols.append(x.cpu().numpy())
        if not pinned:  # a right-hand side's solution does not depend on its place in the batch
            last, _ = c.solve(bt[-1:].contiguous() if batch == 1 else bt.flip(0).contiguous(), p)
            assert torch.equal(last[0], x[-1])
        c.close()
    for j in {0, n - 1}:
        r = b[j] - wilson.apply_m(U, sols[0][j], kappa, -1.0)
        assert np.linalg.norm(r) <= tol * np.linalg.norm(b[j])
    assert np.linalg.norm(sols[0] - sols[1]) <= 1e-9 * np.linalg.norm(sols[1])


@pytest.mark.parametrize("method", [0, 1])
def test_resident_fixed_iterations_and_failures(lib, method):
    """Fixed iterations run exactly that often; NaN, zero and capped right-hand sides are reported as such."""
    dims = (4, 4, 4, 8)
    c = lib.Context(dims)
    c.load_gauge(synthetic.gauge_field(dims, eps=0.45, seed=53))
    c.set_kappa(0.12)
    b = torch.from_numpy(synthetic.random_spinor(dims, seed=54, n=4)).cuda()
    _, st = c.solve(b, lib.Params(precision=1, fixed_iters=9, batch=4, method=method))
    assert [s["iters"] for s in st] == [9] * 4
    b[1] = 0
    b[2].view(-1)[7] = float("nan")
    x, st = c.solve(b, lib.Params(tol=1e-10, precision=1, batch=4, method=method), allow_fail=True)
    assert [s["status"] for s in st] == [0, 0, lib.NAN, 0] and torch.count_nonzero(x[1]).item() == 0
    x, st = c.solve(b[:1].contiguous(), lib.Params(tol=1e-12, precision=1, max_iter=3, batch=4, method=method),
                    allow_fail=True)
    assert st[0]["status"] == lib.NOT_CONVERGED and st[0]["iters"] <= 3
    c.close()
