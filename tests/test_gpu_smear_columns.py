"""Smearing of the non-zero spins only (GPU vs oracle).

Fields with every pattern of vanishing spins, right-hand sides on their own
timeslices (so that groups of columns break in different places), even and odd
numbers of steps (the result ends in either buffer).  Float-float steps: bound
1e-13 of the largest value as for dense fields, and exact zeros stay exact.
"""

import numpy as np
import pytest

import synthetic
from oracle import loops, smear

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def fields(dims, n, seed):
    f = synthetic.random_spinor(dims, seed=seed, n=n)
    for j in range(n):
        for s in range(4):
            if (j >> s) & 1:
                f[j, ..., s, :] = 0.0  # right-hand side j lacks the spins of its bits
    return f


@pytest.mark.parametrize("dims, n, steps", [((4, 4, 4, 4), 17, 5), ((6, 2, 4, 4), 33, 4), ((2, 2, 2, 6), 3, 1)])
def test_smearing_skips_zero_spins(lib, dims, n, steps):
    U = synthetic.gauge_field(dims, eps=0.45, seed=71)
    c = lib.Context(dims)
    c.load_gauge(U)
    eta, phi = fields(dims, n, 72), fields(dims, n, 73)[::-1].copy()
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    ref = smear.smear(U, eta, 3.0, steps)
    got = c.apply_smear(to(eta), 3.0, steps).cpu().numpy()
    assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max()
    for j in range(n):
        for s in range(4):
            if (j >> s) & 1:
                assert not got[j, ..., s, :].any()
    full = loops.smeared_loops(U, eta, phi, 3.0, steps)
    t_of = [(j * j) % dims[3] for j in range(n)]
    got = c.trace_loops(to(eta), to(phi), lib.SINK_SMEARED, smear=(3.0, steps), t_of_rhs=t_of)[:, 0]
    for j in range(n):
        want = np.zeros((16, dims[3]), complex)
        want[:, t_of[j]] = full[j][:, t_of[j]]
        assert np.abs(got[j] - want).max() <= 1e-12 * np.abs(full).max()
    c.close()
