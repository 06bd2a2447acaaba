"""What a user of this library has it do, as measurable cases.

A case is one call, or one short sequence of calls, that a program studying disconnected loops makes through
``paper_1012_5168_gb300.Context`` (or the autograd function built on it), from the smallest lattice to 24^3 x 48:

* ``solve``   M x = b for point or noise sources, in each inner precision and with each Krylov method, with and
              without the clover term;
* ``step``    one noise ensemble: diluted sources, their solves, the local and smeared loops;
* ``exact``   point-source loops on a small lattice;
* ``loops``   local and smeared loops of time-diluted pairs (the sources and solutions are in hand);
* ``mom``     loops at several momenta on all timeslices;
* ``meson``   the connected meson functions of a point source;
* ``grad``    d/dkappa and d/deta of a loop through autograd.

``prepare`` makes seeded SU(3) links U = exp(i eps H) and the fields on the GPU and keeps a Context; ``run`` makes
the call; ``exact`` restates it in 64 bits with plain torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1012_5168_gb300 as dl
from paper_1012_5168_gb300.autograd import loop_trace

PREC = {"f64": dl.PREC_F64, "f32": dl.PREC_F32, "bf16": dl.PREC_BF16}
METHOD = {"bicgstab": dl.METHOD_BICGSTAB, "cgnr": dl.METHOD_CGNR}
DIL24 = dl.DIL_SPIN | dl.DIL_COLOUR | dl.DIL_EVENODD | dl.DIL_TIME
MOMENTA = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
ALPHA, N_SMEAR = 4.0, 50


def _case(kind, dims, n, **more):
    c = dict(kind=kind, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], n=n, batch=32, prec="f32", method="bicgstab",
             kappa=0.14, eps=0.45, csw=0.0, tol=1e-10, source="noise")
    c.update(more)
    return c


def listed():
    p16 = (16, 16, 16, 32)
    return [
        # the ground-truth study: point sources on 4^4, every solve tiny, so that launches and latency count
        dict(_case("exact", (4, 4, 4, 4), 192, batch=64, kappa=0.10, eps=0.30, tol=1e-12), name="exact_4x4x4x4"),
        # one source on the truncated-solver lattice: the smallest solve a program waits for
        dict(_case("solve", (8, 8, 8, 16), 1, batch=1), name="solve_8x8x8x16_single"),
        # CG on the normal equations, the paper's low-precision method, at a batch of 32
        dict(_case("solve", (8, 8, 8, 16), 32, method="cgnr"), name="solve_8x8x8x16_cgnr"),
        # BF16 storage on an uneven lattice with a ragged batch
        dict(_case("solve", (12, 10, 8, 20), 20, prec="bf16", kappa=0.135), name="solve_12x10x8x20_bf16"),
        # the plain double-precision solve of one source on the paper's lattice
        dict(_case("solve", p16, 1, batch=1, prec="f64", tol=1e-11), name="solve_16x16x16x32_f64"),
        # the improved operator, noise sources, the benchmark's width
        dict(_case("solve", p16, 32, kappa=0.13, csw=1.0), name="solve_16x16x16x32_clover"),
        # one propagator (12 point sources, the default batch) on the largest lattice in use
        dict(_case("solve", (24, 24, 24, 48), 12, batch=16, source="point"), name="solve_24x24x24x48_points"),
        # the benchmark's step on two noise vectors: 48 diluted sources, solves, local and smeared loops
        dict(_case("step", p16, 48), name="step_16x16x16x32"),
        # loops of stored pairs on their own timeslices, both sinks
        dict(_case("loops", p16, 48), name="loops_16x16x16x32"),
        # momentum-projected loops of two diluted noise vectors, all timeslices
        dict(_case("mom", p16, 48), name="mom_16x16x16x32"),
        # the pion and all other meson channels from one propagator
        dict(_case("meson", p16, 12), name="meson_16x16x16x32"),
        # loop gradients with respect to kappa and the sources
        dict(_case("grad", (8, 8, 8, 16), 32, tol=1e-12), name="grad_8x8x8x16"),
    ]


def _even(rng, lo, hi):
    return 2 * max(lo // 2, min(hi // 2, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["step", "exact", "loops", "mom", "meson", "grad"])
    while True:
        small = kind in ("exact", "grad")
        hi = 6 if kind == "exact" else (12 if kind == "grad" else 24)
        dims = (_even(rng, 4, hi), _even(rng, 4, hi), _even(rng, 4, hi), _even(rng, 4, 8 if kind == "exact" else (16 if small else 48)))
        V = math.prod(dims)
        n = max(1, round(math.exp(rng.uniform(0.0, math.log(64)))))
        c = _case(kind, dims, n, batch=rng.choice([16, 32, 32, 64]), kappa=round(rng.uniform(0.12, 0.138), 4))
        if kind == "solve":
            c["prec"] = rng.choice(["f32", "f32", "f32", "bf16", "f64"])
            c["tol"] = 1e-11 if c["prec"] == "f64" else 1e-10
            c["source"] = rng.choice(["noise", "noise", "point"])
            c["method"] = rng.choice(["bicgstab"] * 4 + ["cgnr"])
            if c["method"] == "bicgstab" and rng.random() < 0.2:
                c.update(csw=1.0, kappa=round(rng.uniform(0.115, 0.13), 4))
            # double precision issues at a fiftieth of the single-precision rate
            cost = V * n * (12 if c["prec"] == "f64" else 1) * (2 if c["method"] == "cgnr" or c["csw"] else 1)
            if cost > 131072 * 48:
                continue
        elif kind == "exact":
            c.update(n=min(12 * V, 24 * max(1, n // 4)), kappa=0.10, eps=0.30, tol=1e-12)
        elif kind == "grad":
            c.update(n=min(n, 32), tol=1e-12)
        elif kind == "meson":
            c["n"] = 12
        else:
            c["n"] = 24 * max(1, min(2, n // 16))
        if V * c["n"] > 131072 * 48:
            continue
        return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _links(c, seed):
    """SU(3) links exp(i eps H), H = sum_a h_a lambda_a / 2 with Gaussian h: [T][Z][Y][X][4][3][3]."""
    lx, ly, lz, lt = _dims(c)
    h = torch.randn((lt, lz, ly, lx, 4, 8), generator=_gen(seed, 1), device="cuda", dtype=torch.float64) * (0.5 * c["eps"])
    re = torch.zeros(h.shape[:-1] + (3, 3), dtype=torch.float64, device="cuda")
    im = torch.zeros_like(re)
    for a, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        k = (0, 3, 5)[a]  # the symmetric generator of the pair (i, j); the next one is antisymmetric
        re[..., i, j] = re[..., j, i] = h[..., k]
        im[..., i, j], im[..., j, i] = -h[..., k + 1], h[..., k + 1]
    re[..., 0, 0] = h[..., 2] + h[..., 7] / math.sqrt(3)
    re[..., 1, 1] = -h[..., 2] + h[..., 7] / math.sqrt(3)
    re[..., 2, 2] = -2 * h[..., 7] / math.sqrt(3)
    return torch.linalg.matrix_exp(torch.complex(-im, re))  # i H


def _z2(shape, seed, stream):
    s = torch.randint(0, 2, tuple(shape) + (2,), generator=_gen(seed, stream), device="cuda", dtype=torch.int8)
    return torch.view_as_complex((1 - 2 * s).double() * math.sqrt(0.5))


def _times(c, seed):
    """The timeslice of each diluted pair: noise vector m of 24 classes sits on timeslice (m + seed) mod T."""
    return [(int(seed) + j // 24) % c["lt"] for j in range(c["n"])]


def _diluted(c, seed):
    """Spin x colour x even-odd x time diluted Z2 sources, 24 per noise vector."""
    lx, ly, lz, lt = _dims(c)
    eta = torch.zeros((c["n"], lt, lz, ly, lx, 4, 3), dtype=torch.complex128, device="cuda")
    xi = _z2(((c["n"] + 23) // 24, lt, lz, ly, lx, 4, 3), seed, 2)
    z, y, x = torch.meshgrid(torch.arange(lz, device="cuda"), torch.arange(ly, device="cuda"),
                             torch.arange(lx, device="cuda"), indexing="ij")
    for j, t in enumerate(_times(c, seed)):
        k = j % 24
        on = ((x + y + z + t) & 1) == k % 2
        eta[j, t, ..., k // 6, k // 2 % 3] = xi[j // 24, t, ..., k // 6, k // 2 % 3] * on
    return eta


def _sources(c, seed):
    lx, ly, lz, lt = _dims(c)
    shape = (c["n"], lt, lz, ly, lx, 4, 3)
    if c["source"] == "noise":
        return _z2(shape, seed, 2)
    b = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    first = 12 * (int(seed) * 7919 % math.prod(_dims(c)))
    for j in range(c["n"]):
        b[j].view(-1)[(first + j) % b[j].numel()] = 1.0
    return b


def _normal(c, seed, stream):
    lx, ly, lz, lt = _dims(c)
    return torch.randn((c["n"], lt, lz, ly, lx, 4, 3), generator=_gen(seed, stream), device="cuda", dtype=torch.complex128)


def _mom_pair(c, seed):
    """Noise vectors diluted in spin, colour and parity on every timeslice, and solutions of their size."""
    lx, ly, lz, lt = _dims(c)
    eta = torch.zeros((c["n"], lt, lz, ly, lx, 4, 3), dtype=torch.complex128, device="cuda")
    xi = _z2(((c["n"] + 23) // 24, lt, lz, ly, lx, 4, 3), seed, 2)
    t, z, y, x = torch.meshgrid(*(torch.arange(d, device="cuda") for d in (lt, lz, ly, lx)), indexing="ij")
    par = (x + y + z + t) & 1
    for j in range(c["n"]):
        k = j % 24
        eta[j, ..., k // 6, k // 2 % 3] = xi[j // 24, ..., k // 6, k // 2 % 3] * (par == k % 2)
    return eta, eta + 0.3 * _normal(c, seed, 3)


def _context(c, seed):
    ctx = dl.Context(_dims(c), t_bc=-1)
    ctx.load_gauge(_links(c, seed).cpu().numpy())
    ctx.set_kappa(c["kappa"])
    if c["csw"]:
        ctx.set_clover(c["csw"])
    return ctx


def _params(c):
    return dl.Params(tol=c["tol"], precision=PREC[c["prec"]], batch=c["batch"], method=METHOD[c["method"]])


def prepare(c, seed):
    s = dict(c=c, seed=int(seed), ctx=_context(c, seed), p=_params(c))
    kind = c["kind"]
    if kind == "solve":
        s["b"] = _sources(c, seed)
        s["x"] = torch.empty_like(s["b"])
    elif kind == "step":
        s["eta"] = s["ctx"].new_fields(c["n"])
        s["phi"] = s["ctx"].new_fields(c["n"])
        s["t"] = [(int(seed) % 1000 + j // 24) % c["lt"] for j in range(c["n"])]
    elif kind == "loops":
        s["eta"] = _diluted(c, seed)
        s["phi"] = s["eta"] + 0.3 * _normal(c, seed, 3)
        s["t"] = _times(c, seed)
    elif kind == "mom":
        s["eta"], s["phi"] = _mom_pair(c, seed)
    elif kind == "meson":
        s["prop"] = _normal(c, seed, 3)
    elif kind == "grad":
        s["eta"] = _z2(tuple(s["ctx"].new_fields(c["n"]).shape), seed, 2).requires_grad_(True)
        s["kappa"] = torch.tensor(c["kappa"], dtype=torch.float64, requires_grad=True)
    return s


def run(s):
    c, ctx = s["c"], s["ctx"]
    kind = c["kind"]
    if kind == "solve":
        return ctx.solve(s["b"], s["p"], x=s["x"])[0]
    if kind == "step":
        eta = ctx.make_sources(s["seed"], s["seed"] % 1000, c["n"] // 24, DIL24, t0=-1, out=s["eta"])
        phi, _ = ctx.solve(eta, s["p"], x=s["phi"])
        L = ctx.trace_loops(eta, phi, dl.SINK_LOCAL | dl.SINK_SMEARED, smear=(ALPHA, N_SMEAR), t_of_rhs=s["t"], group=24)
        return {"phi": phi, "loops": L}
    if kind == "exact":
        return ctx.exact_loops(0, c["n"], s["p"])[0]
    if kind == "loops":
        return ctx.trace_loops(s["eta"], s["phi"], dl.SINK_LOCAL | dl.SINK_SMEARED, smear=(ALPHA, N_SMEAR),
                               t_of_rhs=s["t"], group=24)
    if kind == "mom":
        return ctx.trace_loops_mom(s["eta"], s["phi"], MOMENTA, dl.SINK_LOCAL, group=24)
    if kind == "meson":
        return ctx.meson_correlators(s["prop"], (0, 0, 0, 0), MOMENTA)
    L = loop_trace(s["eta"], s["kappa"], ctx, s["p"])
    g = torch.autograd.grad(L[:, 5].real.sum(), [s["eta"], s["kappa"]])
    return {"loops": L.detach(), "eta": g[0], "kappa": g[1]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(c):
    V, n = math.prod(_dims(c)), c["n"]
    V3 = V // c["lt"]
    field, links = V * 192, V * 576
    # BiCGStab iterations of the even-odd system at this kappa, two matrix products of two half hops each
    iters = math.log(1.0 / c["tol"]) * 0.25 / (1.0 - c["kappa"] / 0.148)
    solve = n * V * (1320.0 + 100.0) * 2 * iters
    kind = c["kind"]
    if kind == "solve":
        return dict(bytes=2 * n * field + links, flops=solve)
    if kind == "exact":
        return dict(bytes=links + 256 * c["lt"], flops=solve)
    if kind == "grad":
        return dict(bytes=2 * n * field + links, flops=2 * solve)
    # per pair and iteration of smearing: six directions, four spins, a 3 x 3 complex product, both fields
    smear = n * V3 * N_SMEAR * 2 * 6 * 4 * 66.0
    if kind == "step":
        return dict(bytes=2 * n * field + links, flops=solve + smear)
    if kind == "loops":
        return dict(bytes=2 * n * V3 * 192 + links, flops=smear + 2 * n * V3 * 384)
    if kind == "mom":
        return dict(bytes=2 * n * field, flops=n * V * 48 * 8.0)
    return dict(bytes=12 * field, flops=V * 136 * 9 * 8.0 + V * 136 * len(MOMENTA) * 8.0)


# ---------------------------------------------------------------------------
# the same in 64 bits: plain torch, fields [T][Z][Y][X][3][4][n]
# ---------------------------------------------------------------------------
def _gammas():
    """The 16 matrices 1, g_mu, g5, g5 g_mu, g_mu g_nu (mu < nu) of the chiral basis."""
    i = 1j
    g = [np.array(m, dtype=complex) for m in (
        [[0, 0, 0, i], [0, 0, i, 0], [0, -i, 0, 0], [-i, 0, 0, 0]], [[0, 0, 0, -1], [0, 0, 1, 0], [0, 1, 0, 0], [-1, 0, 0, 0]],
        [[0, 0, i, 0], [0, 0, 0, -i], [-i, 0, 0, 0], [0, i, 0, 0]], [[0, 0, 1, 0], [0, 0, 0, 1], [1, 0, 0, 0], [0, 1, 0, 0]])]
    g5 = g[0] @ g[1] @ g[2] @ g[3]
    out = [np.eye(4, dtype=complex)] + g + [g5] + [g5 @ m for m in g] + [g[a] @ g[b] for a in range(4) for b in range(a + 1, 4)]
    return torch.from_numpy(np.stack(out)).cuda()


def _inner(v):
    return v.permute(1, 2, 3, 4, 6, 5, 0).contiguous()


def _outer(v):
    return v.permute(6, 0, 1, 2, 3, 5, 4).contiguous()


def _mm(u, h):
    return torch.matmul(u, h.flatten(-2)).view(h.shape)


def _clover(U, kappa, csw):
    """A = 1 - kappa csw sum sigma F as [T][Z][Y][X][12][12] (colour slow, spin fast)."""
    G = _gammas()
    ax = (3, 2, 1, 0)
    dag = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
    A = torch.eye(12, dtype=torch.complex128, device="cuda").expand(U.shape[:4] + (12, 12)).clone()
    for m in range(4):
        for n in range(m + 1, 4):
            a, b = U[..., m, :, :], U[..., n, :, :]
            at = lambda v, dm, dn: v.roll(-dm, ax[m]).roll(-dn, ax[n])  # noqa: E731
            q = a @ at(b, 1, 0) @ dag(at(a, 0, 1)) @ dag(b)
            q = q + b @ dag(at(a, -1, 1)) @ dag(at(b, -1, 0)) @ at(a, -1, 0)
            q = q + dag(at(a, -1, 0)) @ dag(at(b, -1, -1)) @ at(a, -1, -1) @ at(b, 0, -1)
            q = q + dag(at(b, 0, -1)) @ at(a, 0, -1) @ at(b, 1, -1) @ dag(a)
            F = (q - dag(q)) / 8j
            sig = 0.5j * (G[1 + m] @ G[1 + n] - G[1 + n] @ G[1 + m])
            A -= kappa * csw * torch.einsum("...ab,st->...asbt", F, sig).reshape(A.shape)
    return A


class _Wilson:
    """M = A - kappa D on fields [T][Z][Y][X][3][4][n] in the type of the links."""

    def __init__(self, U, kappa, csw):
        self.k = kappa
        self.u = [U[..., m, :, :].contiguous() for m in range(4)]
        self.u[3] = self.u[3].clone()
        self.u[3][-1] *= -1  # antiperiodic in time
        self.ud = [u.conj().transpose(-1, -2).contiguous() for u in self.u]
        self.A = None
        ph = lambda a, b: torch.tensor([[a], [b]], dtype=U.dtype, device="cuda")  # noqa: E731
        self.X = [(True, ph(1j, 1j)), (True, ph(-1, 1)), (False, ph(1j, -1j)), (False, ph(1, 1))]
        if csw:
            self.A = _clover(U.to(torch.complex128), kappa, csw).to(U.dtype)

    def low(self):
        m = object.__new__(_Wilson)
        to = lambda v: v.to(torch.complex64)  # noqa: E731
        m.k, m.u, m.ud = self.k, [to(v) for v in self.u], [to(v) for v in self.ud]
        m.A = to(self.A) if self.A is not None else None
        m.X = [(f, to(p)) for f, p in self.X]
        return m

    def hop(self, v):
        out = torch.zeros_like(v)
        for m in range(4):
            flip, ph = self.X[m]
            ax = 3 - m
            for s in (-1, 1):
                src = v.roll(-1, ax) if s < 0 else v
                d = src[..., 2:, :].flip(-2) if flip else src[..., 2:, :]
                h = src[..., :2, :] + s * ph * d
                w = _mm(self.u[m], h) if s < 0 else _mm(self.ud[m], h).roll(1, ax)
                out[..., :2, :] += w
                e = ph.conj() * w
                out[..., 2:, :] += s * (e.flip(-2) if flip else e)  # s X^dag w
        return out

    def __call__(self, v):
        a = v if self.A is None else torch.matmul(self.A, v.flatten(-3, -2)).view(v.shape)
        return a - self.k * self.hop(v)


def _dots(a, b):
    return (a.conj() * b).sum(dim=tuple(range(6)), dtype=torch.complex128)


def _solve64(M, b, dagger=False):
    """x with |b - M x| <= 1e-13 |b|: BiCGStab in single precision under double-precision refinement."""
    if dagger:  # M^dag = g5 M g5
        g5 = torch.tensor([1, 1, -1, -1], dtype=torch.float64, device="cuda").view(4, 1)
        return g5 * _solve64(M, g5 * b)
    m = M.low()
    x = torch.zeros_like(b)
    b2 = _dots(b, b).real
    for _ in range(8):
        r64 = b - M(x)
        nrm = _dots(r64, r64).real.sqrt()
        if float((nrm / b2.sqrt()).max()) < 1e-13:
            break
        r = (r64 / nrm.clamp_min(1e-300)).to(torch.complex64)
        e, rh, p = torch.zeros_like(r), m(m(r)), r.clone()  # (a point source is its own shadow's breakdown)
        rho = _dots(rh, r)
        for it in range(600):
            v = m(p)
            on = _dots(r, r).real > 1e-11  # a column that is done stays as it is
            al = torch.where(on, rho / _dots(rh, v), 0).to(r.dtype)
            s = r - al * v
            t = m(s)
            om = torch.where(on, _dots(t, s) / _dots(t, t).real.clamp_min(1e-30), 0).to(r.dtype)
            e += al * p + om * s
            r = s - om * t
            new = _dots(rh, r)
            p = r + torch.where(on, (new / rho) * (al / om), 0).to(r.dtype) * (p - om * v)
            rho = torch.where(on, new, rho)
            if it % 4 == 3 and float(_dots(r, r).real.max()) < 1e-9:
                break
        x = x + nrm * e.to(torch.complex128)
    return x


def _loops(eta, phi):
    """[n][16][T] of canonical fields."""
    return torch.einsum("gab,ntab->ngt", _gammas(), torch.einsum("ntzyxac,ntzyxbc->ntab", eta.conj(), phi))


def _smear(U3, v):
    """K of canonical single-timeslice fields [n][Z][Y][X][4][3] on the timeslice's links."""
    v = v.permute(1, 2, 3, 5, 4, 0).contiguous()
    for _ in range(N_SMEAR):
        h = torch.zeros_like(v)
        for m in range(3):
            u, ax = U3[..., m, :, :], 2 - m
            h += _mm(u, v.roll(-1, ax)) + _mm(u.conj().transpose(-1, -2), v).roll(1, ax)
        v = (v + ALPHA * h) / (1 + 6 * ALPHA)
    return v.permute(5, 0, 1, 2, 4, 3)


def _traced(c, U, eta, phi, times):
    """[n / 24][2 sinks][16][T]: the loops of each pair on its timeslice, 24 pairs summed."""
    out = torch.zeros((c["n"] // 24, 2, 16, c["lt"]), dtype=torch.complex128, device="cuda")
    for g in range(c["n"] // 24):
        t, j = times[24 * g], slice(24 * g, 24 * g + 24)
        for s, (e, f) in enumerate(((eta[j, t], phi[j, t]), (_smear(U[t], eta[j, t]), _smear(U[t], phi[j, t])))):
            out[g, s, :, t] = _loops(e[:, None], f[:, None]).sum(0)[:, 0]
    return out


def _philox_sources(c, seed, first):
    """make_sources of the step case: signs of Philox4x64-10 with key (seed, 0), counter (site / 4, noise, 0, 0)."""
    lx, ly, lz, lt = _dims(c)
    V = math.prod(_dims(c))
    eta = torch.zeros((c["n"], lt, lz, ly, lx, 4, 3), dtype=torch.complex128, device="cuda")
    z, y, x = torch.meshgrid(torch.arange(lz), torch.arange(ly), torch.arange(lx), indexing="ij")
    for m in range(c["n"] // 24):
        noise, t = first + m, (first + m) % lt
        start = ((noise << 64) - 1) % (1 << 256)  # the generator advances its counter before each block
        words = np.array([(start >> (64 * k)) & (2**64 - 1) for k in range(4)], dtype=np.uint64)
        raw = np.random.Philox(key=np.array([seed, 0], dtype=np.uint64), counter=words).random_raw(V)
        w = torch.from_numpy(raw.reshape(lt, lz, ly, lx)[t].astype(np.int64))
        for k in range(24):
            sc = 3 * (k // 6) + k // 2 % 3
            sign = [(1 - 2 * ((w >> (2 * sc + q)) & 1)).double() for q in (0, 1)]
            on = ((x + y + z + t) & 1) == k % 2
            eta[24 * m + k, t, ..., k // 6, k // 2 % 3] = (torch.complex(*sign) * math.sqrt(0.5) * on).cuda()
    return eta


def exact(c, seed):
    torch.backends.cuda.matmul.allow_tf32 = False
    kind, V = c["kind"], math.prod(_dims(c))
    lx, ly, lz, lt = _dims(c)
    G = _gammas()
    if kind == "meson":
        S = _normal(c, seed, 3).view(4, 3, lt, lz * ly * lx, 4, 3)  # [alpha][a][t][site][beta][b]
        g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")
        out = torch.zeros((len(MOMENTA), 16, 16, lt), dtype=torch.complex128, device="cuda")
        for t in range(lt):
            P = torch.einsum("iaxbc,jaxdc->xbidj", S[:, :, t].conj(), S[:, :, t])
            F = torch.einsum("qx,xbidj->qbidj", _phases(c), P)
            out[..., t] = -torch.einsum("i,b,Bbd,Aji,qbidj->qAB", g5.to(P.dtype), g5.to(P.dtype), G, G, F)
        return out.cpu().numpy()
    if kind == "mom":
        eta, phi = _mom_pair(c, seed)
        out = []
        for g in range(c["n"] // 24):
            S = sum(torch.einsum("txac,txbc->txab", eta[j].view(lt, -1, 4, 3).conj(), phi[j].view(lt, -1, 4, 3))
                    for j in range(24 * g, 24 * g + 24))
            out.append(torch.einsum("gab,qx,txab->qgt", G, _phases(c), S))
        return torch.stack(out)[:, None].cpu().numpy()
    if V * c["n"] * (2 if kind == "grad" else 1) > 131072 * 49:
        return None
    U = _links(c, seed)
    if kind == "loops":
        eta = _diluted(c, seed)
        return _traced(c, U, eta, eta + 0.3 * _normal(c, seed, 3), _times(c, seed)).cpu().numpy()
    M = _Wilson(U, c["kappa"], c["csw"])

    def solve(b, **kw):
        return torch.cat([_outer(_solve64(M, _inner(b[j:j + 16]), **kw)) for j in range(0, len(b), 16)])

    if kind == "solve":
        return solve(_sources(c, seed))
    if kind == "step":
        first = int(seed) % 1000
        eta = _philox_sources(c, int(seed), first)
        phi = solve(eta)
        times = [(first + j // 24) % lt for j in range(c["n"])]
        return {"phi": phi, "loops": _traced(c, U, eta, phi, times).cpu().numpy()}
    if kind == "exact":
        out = torch.zeros((1, 16, lt), dtype=torch.complex128, device="cuda")
        for j0 in range(0, c["n"], 48):
            js = range(j0, min(c["n"], j0 + 48))
            b = torch.zeros((len(js), lt, lz, ly, lx, 4, 3), dtype=torch.complex128, device="cuda")
            for k, j in enumerate(js):
                b[k].view(-1)[j] = 1.0
            x = solve(b).view(len(js), V, 4, 3)
            for k, j in enumerate(js):
                i, al, a = j // 12, j // 3 % 4, j % 3
                out[0, :, i // (V // lt)] += torch.einsum("gb,b->g", G[:, al], x[k, i, :, a])
        return out.cpu().numpy()
    eta = _z2((c["n"], lt, lz, ly, lx, 4, 3), seed, 2)
    phi = solve(eta)
    L = _loops(eta, phi)
    g5 = G[5].diagonal().real.view(4, 1)
    chi = solve(g5 * eta, dagger=True)
    dphi = _outer(M.hop(_inner(phi)))
    return {"loops": L, "eta": chi + g5 * phi, "kappa": (chi.conj() * dphi).sum().real.cpu()}


def _phases(c):
    """exp(-i p.x) of the listed momenta: [momentum][Z Y X]."""
    lx, ly, lz, _ = _dims(c)
    z, y, x = torch.meshgrid(*(torch.arange(d, device="cuda", dtype=torch.float64) / d for d in (lz, ly, lx)), indexing="ij")
    return torch.stack([torch.exp(-2j * math.pi * (m[0] * x + m[1] * y + m[2] * z)).reshape(-1) for m in MOMENTA])
