"""Momentum loops and meson functions with many momenta, and groups whose pairs several blocks share (GPU vs oracle).

Momentum lists whose representatives leave remainders of 1, 2 and 3 against the four of a warp, zero momentum
alone, first, and as the last and only one of its four; timeslices of 128 sites on 16 timeslices (64 blocks for
one group: its pairs go to three) and of 8 sites (one pair a block).  Bound: FP64 sums of at most 12 x 128 x 3
products, 1e-12 of the largest value.
"""

import itertools

import numpy as np
import pytest

import synthetic
from oracle import correlators, lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MANY = list(itertools.product(range(-1, 2), range(-1, 2), range(0, 2))) + [(0, 0, 3)]
LISTS = [[(0, 0, 0)], [(0, 0, 0), (1, 0, 0)], [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 0, 0)],
         [(1, 0, 0), (-1, 0, 0), (0, 1, 1), (9, 0, 0), (0, -1, -1), (0, 0, 2), (1, 1, 1)], MANY]


@pytest.mark.parametrize("dims", [(8, 4, 4, 16), (2, 2, 2, 4)])
@pytest.mark.parametrize("moms", LISTS)
def test_momentum_lists_and_shared_groups(lib, dims, moms):
    G = lattice.gamma_basis()
    eta, phi = (synthetic.random_spinor(dims, seed=s, n=12) for s in (65, 66))
    c = lib.Context(dims)
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    ref = correlators.momentum_loops(eta, phi, moms, G)
    for group in (12, 6, 4, 1):
        want = ref.reshape(12 // group, group, *ref.shape[1:]).sum(1)
        got = c.trace_loops_mom(to(eta), to(phi), moms, group=group)[:, 0]
        assert np.abs(got - want).max() < 1e-12 * np.abs(ref).max() * group
    t_of = [3] * 12
    got = c.trace_loops_mom(to(eta), to(phi), moms, t_of_rhs=t_of, group=12)[:, 0]
    want = np.zeros_like(ref[:1])
    want[0, ..., 3] = ref[..., 3].sum(0)
    assert np.abs(got - want).max() < 1e-12 * np.abs(ref).max() * 12
    if dims[3] != 4:
        return c.close()  # (the oracle's meson functions take too long there)
    src = (1, 0, 1, 2)
    ref = correlators.connected(phi, src, moms, G)
    assert np.abs(c.meson_correlators(to(phi), src, moms) - ref).max() < 1e-12 * np.abs(ref).max()
    c.close()
