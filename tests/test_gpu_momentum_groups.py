"""Momentum loops summed over groups at the sites, and meson functions from the hermitian half (GPU vs oracle).

Sizes at the edges of the kernels: timeslices of 8, 48 and 64 sites against tiles
of 32, rows of 2 to 8 sites, groups of 1, 3 and 6 pairs, groups whose pairs sit on
one or on several timeslices, fields that vanish in whole spins, colours and
parities, and momentum lists with p, -p, equal and wrapped entries.  Bound: FP64
sums of at most 6 x 48 products, 1e-12 of the largest loop.
"""

import numpy as np
import pytest

import synthetic
from oracle import correlators, lattice, noise

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MOMS = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, -1), (0, -1, 1), (1, 0, 0), (7, 0, 1), (0, 0, -2), (1, 1, 1)]


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (6, 2, 4, 6), (4, 4, 4, 4), (8, 2, 4, 2)])
@pytest.mark.parametrize("group, spread", [(1, False), (6, False), (3, True), (6, True)])
def test_grouped_momentum_loops(lib, dims, group, spread):
    G = lattice.gamma_basis()
    T = dims[3]
    eta = noise.make_sources(dims, 3, 0, 1, noise.SPIN | noise.COLOUR)[:12]
    eta[6:] += synthetic.random_spinor(dims, seed=61, n=6)  # half of them diluted, half dense
    phi = synthetic.random_spinor(dims, seed=62, n=12)
    c = lib.Context(dims)
    c.load_gauge(synthetic.gauge_field(dims, eps=0.4, seed=63))
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    t_of = [(j if spread else j // 6) % T for j in range(12)]
    ref = correlators.momentum_loops(eta, phi, MOMS, G)  # [12][Q][16][T]
    scale = np.abs(ref).max()
    got = c.trace_loops_mom(to(eta), to(phi), MOMS, group=group)[:, 0]
    assert np.abs(got - ref.reshape(12 // group, group, *ref.shape[1:]).sum(1)).max() < 1e-12 * scale * group
    one = np.zeros_like(ref)
    for j in range(12):
        one[j, ..., t_of[j]] = ref[j, ..., t_of[j]]
    got = c.trace_loops_mom(to(eta), to(phi), MOMS, lib.SINK_LOCAL | lib.SINK_SMEARED, smear=(2.0, 0), t_of_rhs=t_of,
                            group=group)
    want = one.reshape(12 // group, group, *ref.shape[1:]).sum(1)
    for s in range(2):  # (no smearing steps: both sinks are the local one, through canonical and converted fields)
        assert np.abs(got[:, s] - want).max() < 1e-12 * scale * group
    bad = phi.copy()
    bad[0, 1, 0, 0, 1, 3, 2] = np.nan  # eta[0] is zero in spin 3
    got = c.trace_loops_mom(to(eta), to(bad), MOMS, group=group)[:, 0]
    assert np.isnan(got[0][:, 0, 1]).all() and np.isfinite(got[0][:, :, 0]).all()
    c.close()


@pytest.mark.parametrize("dims, src", [((2, 2, 2, 4), (1, 0, 1, 3)), ((6, 2, 4, 2), (5, 1, 2, 0))])
def test_meson_from_hermitian_half(lib, dims, src):
    G = lattice.gamma_basis()
    prop = synthetic.random_spinor(dims, seed=64, n=12)
    c = lib.Context(dims)
    got = c.meson_correlators(torch.from_numpy(prop).cuda(), src, MOMS)
    ref = correlators.connected(prop, src, MOMS, G)
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()
    c.close()
