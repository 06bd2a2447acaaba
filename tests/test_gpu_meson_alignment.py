"""Meson functions of a propagator that starts on an 8-byte boundary (GPU vs oracle).

The C interface takes a pointer to doubles; one past the start of an allocation is no 16-byte boundary.
Bound: FP64 sums of 9 x 48 products, 1e-12 of the largest value; both reads add in the same order.
"""

import ctypes

import numpy as np
import pytest

import synthetic
from oracle import correlators, lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MOMS = [(0, 0, 0), (1, 0, 0), (-1, 0, 0)]


@pytest.mark.parametrize("dims", [(2, 2, 2, 4), (6, 2, 4, 2)])
def test_propagator_on_an_eight_byte_boundary(lib, dims):
    prop = synthetic.random_spinor(dims, seed=64, n=12)
    c = lib.Context(dims)
    aligned = c.meson_correlators(torch.from_numpy(prop).cuda(), (1, 0, 1, 1), MOMS)
    buf = torch.empty(prop.size * 2 + 1, dtype=torch.float64, device="cuda")
    buf[1:] = torch.from_numpy(prop.view(np.float64).ravel()).cuda()
    torch.cuda.synchronize()
    assert (buf.data_ptr() + 8) % 16 == 8
    out = np.empty((len(MOMS), 16, 16, dims[3]), dtype=np.complex128)
    mom = np.asarray(MOMS, dtype=np.int32)
    rc = lib.lib().dl_meson_correlators(c._h, ctypes.c_void_p(buf.data_ptr() + 8), (ctypes.c_int * 4)(1, 0, 1, 1),
                                        mom.ctypes.data_as(ctypes.POINTER(ctypes.c_int)), len(MOMS),
                                        out.ctypes.data_as(ctypes.c_void_p))
    assert rc == 0
    ref = correlators.connected(prop, (1, 0, 1, 1), MOMS, lattice.gamma_basis())
    assert np.abs(out - ref).max() < 1e-12 * np.abs(ref).max()
    assert np.array_equal(out, aligned)
    c.close()
