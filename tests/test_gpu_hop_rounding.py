"""Rounding of the FP64 Wilson hop against extended precision (GPU).

Reference order: every product U h and U^dag h in its own FMA chain over the colours, added to the spins one
after the other (forward, backward, mu = 0 .. 3).  The kernels may add in another order, but no carried value
may lose more bits: the root mean square error has to stay within the reference order's (2% for the sampling
error, which is 1 / sqrt(2 x 196,608 values) = 0.2% a side).  All three whole-hop sizes run: four warps to 32
sites in one group and in two, and the whole-site kernel.
"""

import numpy as np
import pytest

import synthetic
from oracle import wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

L = np.longdouble


def _fma(a, b, c):  # one rounding: the extended product and sum are exact to 2^-64 or better
    return (a.astype(L) * b + c).astype(np.float64)


def _parts(z):
    return z.real.copy(), z.imag.copy()


def _neighbours(U, psi):
    """(links [sites][3][3], projected half spinors, s X^dag) of the eight directions, in the kernel's order."""
    X = (np.array([[0, 1j], [1j, 0]]), np.array([[0, -1], [1, 0]]), np.array([[1j, 0], [0, -1j]]), np.eye(2))
    for mu in range(4):
        u = U[..., mu, :, :]
        back = np.roll(u, 1, axis=wilson.site_axis(mu)).conj().swapaxes(-1, -2)
        for s, link, q in ((-1, u, wilson._shift_forward(psi, mu, -1.0)), (+1, back, wilson._shift_backward(psi, mu, -1.0))):
            h = q[..., :2, :] + s * np.einsum("st,...ta->...sa", X[mu], q[..., 2:, :])  # (one FP64 addition each)
            yield link, h, s * X[mu].conj().T


def _reference_order(U, psi):
    acc = np.zeros(psi.shape, dtype=np.complex128)
    for link, h, xd in _neighbours(U, psi):
        ur, ui = _parts(link)
        hr, hi = _parts(h)
        wr, wi = np.zeros_like(hr), np.zeros_like(hi)
        for b in range(3):
            r, i = ur[..., None, :, b], ui[..., None, :, b]
            x, y = hr[..., b, None], hi[..., b, None]
            wr = _fma(-i, y, _fma(r, x, wr))
            wi = _fma(i, x, _fma(r, y, wi))
        w = wr + 1j * wi
        acc[..., :2, :] += w
        acc[..., 2:, :] += np.einsum("st,...ta->...sa", xd, w)  # (phases: exact)
    return acc


def _extended(U, psi):
    acc = np.zeros(psi.shape, dtype=np.clongdouble)
    X = (np.array([[0, 1j], [1j, 0]]), np.array([[0, -1], [1, 0]]), np.array([[1j, 0], [0, -1j]]), np.eye(2))
    p = psi.astype(np.clongdouble)
    for mu in range(4):
        u = U[..., mu, :, :]
        back = np.roll(u, 1, axis=wilson.site_axis(mu)).conj().swapaxes(-1, -2)
        for s, link, q in ((-1, u, wilson._shift_forward(p, mu, -1.0)), (+1, back, wilson._shift_backward(p, mu, -1.0))):
            h = q[..., :2, :].copy()
            for a in range(2):
                for b in range(2):
                    h[..., a, :] += s * X[mu][a, b] * q[..., 2 + b, :]
            w = np.zeros_like(h)
            for b in range(3):
                w += link.astype(np.clongdouble)[..., None, :, b] * h[..., b, None]
            acc[..., :2, :] += w
            for a in range(2):
                for b in range(2):
                    acc[..., 2 + a, :] += s * X[mu].conj().T[a, b] * w[..., b, :]
    return acc


@pytest.mark.parametrize("dims, n", [((4, 4, 4, 8), 16), ((4, 4, 8, 16), 4), ((8, 8, 8, 16), 1), ((8, 8, 8, 4), 64)])
def test_hop_error_within_the_reference_order(lib, dims, n):
    U = synthetic.gauge_field(dims, eps=0.45, seed=97)
    psi = synthetic.random_spinor(dims, seed=98, n=n)
    m = min(n, 16)
    exact = _extended(U, psi[:m])
    rms = lambda v: float(np.sqrt((np.abs((v - exact).astype(np.complex128)) ** 2).mean()))  # noqa: E731
    want = rms(_reference_order(U, psi[:m]))
    c = lib.Context(dims)
    c.load_gauge(U)
    c.set_kappa(0.1)
    got = rms(c.apply_hop(torch.from_numpy(psi).cuda()).cpu().numpy()[:m])
    assert got <= 1.02 * want
    c.close()
