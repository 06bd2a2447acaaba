"""The FP64 quotients of the Krylov recurrences against CUDA's division, and solves driven to underflow (GPU).

``fp64_rcp`` is within 2^-52 of 1/x over its range; a product with it adds one rounding, so a quotient is within
2^-51 of CUDA's correctly rounded one.  Outside that range (subnormal and huge divisors, zero, infinities,
NaN) the quotients are CUDA's, bit by bit.
"""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r"""
#include "launch.h"
namespace {
__global__ void quotients(const double *a, const double *b, int n, double *out, double *ref) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = dl::fp64_div(a[i], b[i]);
    const double2 q = dl::fp64_div(make_double2(a[i], -a[i]), b[i]);
    out[n + i] = q.x;
    out[2 * n + i] = -q.y;
    ref[i] = a[i] / b[i];
}
}
extern "C" int run(const double *a, const double *b, int n, double *out, double *ref) {
    quotients<<<(n + 127) / 128, 128>>>(a, b, n, out, ref);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def quotients(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    from paper_1012_5168_gb300 import build
    d = tmp_path_factory.mktemp("quotients")
    src, so = d / "quotients.cu", d / "quotients.so"
    src.write_text(SOURCE)
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-shared", "-o", str(so), str(src)], check=True)
    fn = ctypes.CDLL(str(so)).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def call(a, b):
        x, y = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        out = torch.empty((3, len(a)), dtype=torch.float64, device="cuda")
        ref = torch.empty(len(a), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(x.data_ptr(), y.data_ptr(), len(a), out.data_ptr(), ref.data_ptr()) == 0
        return out.cpu().numpy(), ref.cpu().numpy()
    return call


def test_quotients_over_all_exponents(quotients):
    rng = np.random.default_rng(5)
    e = np.repeat(np.arange(-1074, 1024), 64)
    b = np.ldexp(1.0 + rng.random(e.size), e) * rng.choice([-1.0, 1.0], e.size)
    for a in (np.ones(e.size), np.ldexp(1.0 + rng.random(e.size), np.clip(e + rng.integers(-30, 30, e.size), -1022, 1023))):
        out, ref = quotients(a, b)
        inside = (np.abs(b) >= np.ldexp(1.0, -1020)) & (np.abs(b) < np.ldexp(1.0, 1020))
        assert np.array_equal(out[:, ~inside], np.broadcast_to(ref[~inside], (3, (~inside).sum())))
        ok = inside & (np.abs(ref) > np.ldexp(1.0, -1000))  # (a subnormal quotient has fewer bits)
        assert ok.sum() > 64 * 2000
        assert (np.abs(out[:, ok] - ref[ok]) <= np.ldexp(np.abs(ref[ok]), -51)).all()


def test_quotients_of_special_values(quotients):
    v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1e308, 1.0])
    a, b = (m.ravel().copy() for m in np.meshgrid(v, v))
    out, ref = quotients(a, b)
    special = ~((b == 1.0) & np.isfinite(a))
    for row in out:
        assert np.array_equal(row[special], ref[special], equal_nan=True) and np.array_equal(row[~special], a[~special])


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 2, 4)])
@pytest.mark.parametrize("method", [0, 1])
def test_iterations_past_convergence_stay_finite(lib, dims, method):
    """Fixed iterations go on until the recurrence's residual underflows; the solution is not touched by that."""
    U = synthetic.gauge_field(dims, eps=0.45, seed=60)
    b = torch.from_numpy(synthetic.random_spinor(dims, seed=61, n=16)).cuda()
    for prec in (0, 1):
        for kappa in (0.01, 0.02, 0.025, 0.03, 0.04, 0.08):
            c = lib.Context(dims)
            c.load_gauge(U)
            c.set_kappa(kappa)
            for iters in (40, 400):
                x, st = c.solve(b, lib.Params(precision=prec, fixed_iters=iters, batch=16, method=method), allow_fail=True)
                assert torch.isfinite(torch.view_as_real(x)).all(), (kappa, iters, st)
                r = b - c.apply_m(x)
                tol = 1e-12 if prec == 0 else 1e-5  # one inner phase: 53 and 24 bits, 500 and 80 roundings to spare
                assert (r.flatten(1).norm(dim=1) <= tol * b.flatten(1).norm(dim=1)).all()
            c.close()
