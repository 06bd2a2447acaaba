"""Smearing on both sides of the sizes where its columns are listed and its list is spread (GPU vs oracle).

Launches of 256 threads over (site, colour row, right-hand side, field) that give 152 SMs at most one block, up
to two, and more, with every pattern of vanishing spins; each context smears twice, so that what one smearing
leaves behind would show in the next.  Float-float steps: bound 1e-13 of the largest value.
"""

import numpy as np
import pytest

import synthetic
from oracle import loops, smear

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def fields(dims, n, seed, shift):
    f = synthetic.random_spinor(dims, seed=seed, n=n)
    for j in range(n):
        for s in range(4):
            if ((j + shift) >> s) & 1:
                f[j, ..., s, :] = 0.0  # right-hand side j lacks the spins of the bits of j + shift
    return f


@pytest.mark.parametrize("dims, n, steps", [((4, 4, 4, 2), 20, 3), ((8, 8, 8, 2), 17, 3), ((8, 8, 8, 2), 34, 2),
                                            ((8, 6, 8, 4), 17, 3), ((10, 10, 10, 2), 34, 3)])
def test_smearing_with_and_without_a_list(lib, dims, n, steps):
    U = synthetic.gauge_field(dims, eps=0.45, seed=74)
    c = lib.Context(dims)
    c.load_gauge(U)
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    for shift in (0, 5):
        eta, phi = fields(dims, n, 75, shift), fields(dims, n, 76, 2 * shift)[::-1].copy()
        ref = smear.smear(U, eta, 3.0, steps)
        got = c.apply_smear(to(eta), 3.0, steps).cpu().numpy()
        assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max()
        for j in range(n):
            for s in range(4):
                if ((j + shift) >> s) & 1:
                    assert not got[j, ..., s, :].any()
        full = loops.smeared_loops(U, eta, phi, 3.0, steps)
        # timeslices that change from pair to pair, and in runs of 17 (for those the columns are listed)
        for t_of in ([(j * j + shift) % dims[3] for j in range(n)], [(j // 17 + shift) % dims[3] for j in range(n)]):
            got = c.trace_loops(to(eta), to(phi), lib.SINK_SMEARED, smear=(3.0, steps), t_of_rhs=t_of)[:, 0]
            for j in range(n):
                want = np.zeros((16, dims[3]), complex)
                want[:, t_of[j]] = full[j][:, t_of[j]]
                assert np.abs(got[j] - want).max() <= 1e-12 * np.abs(full).max()
    c.close()
