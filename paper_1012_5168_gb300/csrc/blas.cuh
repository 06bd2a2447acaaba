// BiCGStab vector updates, scalar recurrences and the FP64 defect-correction
// steps, for N right-hand sides in the even-odd tile layout (see common.cuh).
//
// The Krylov solver is BiCGStab (van der Vorst 1992; Sec. 2 of the paper uses
// QUDA's mixed-precision CG/BiCGStab) on the even-site Schur complement
// Mhat = 1 - kappa^2 D_eo D_oe.  One iteration, per right-hand side:
//
//   v = Mhat p                 (two hops; <rhat, v> fused in the second)
//   alpha = rho / <rhat, v>
//   s = r - alpha v
//   t = Mhat s                 (two hops; <t,s>, <t,t>, <rhat,s>, <rhat,t>, <s,s> fused)
//   omega = <t,s> / <t,t>
//   rho'  = <rhat, s - omega t> = <rhat,s> - omega <rhat,t>
//   beta  = (rho'/rho) (alpha/omega)
//   |r'|^2 = <s,s> - |<t,s>|^2/<t,t>      (r' = s - omega t)
//   x += alpha p + omega s ;  r = s - omega t ;  p = r + beta (p - omega v)
//
// Knowing rho' and beta before the vector update lets one kernel do all three
// updates (5 reads, 3 writes per element).  Per-right-hand-side scalars live in
// device memory (RhsState) so whole iterations can be captured in CUDA graphs;
// every right-hand side carries its own active flag and stops independently.
#pragma once

#include "common.cuh"

namespace dl {

enum { ST_OK = 0, ST_BREAKDOWN = 5, ST_NAN = 6 };

struct RhsState {
    double2 rho, alpha, omega, beta;
    double r2;       // recursive residual norm^2 of the inner iteration
    double r2_0;     // at the start of the inner cycle
    double target2;  // stop the inner cycle when r2 <= target2
    int active;      // takes part in the current iteration
    int next_active; // takes part in the next iteration
    int iters;       // inner iterations in this cycle
    int status;      // ST_OK / ST_BREAKDOWN / ST_NAN (inner cycle)
    int max_iters;   // cap on iterations in this cycle
    int fixed;       // 1: run exactly max_iters iterations
};

struct OuterState {
    double b2;        // |bhat|^2 (even-site Schur system)
    double r2;        // |bhat - Mhat x|^2 (FP64 true residual of the Schur system)
    double full_b2;   // |b|^2 (full lattice)
    double full_r2;   // |b - M x|^2 (full lattice)
    double tol2;      // tol^2
    int active;       // not yet converged
    int status;
    int outer;        // defect-correction cycles done
    int iters;        // inner iterations summed over cycles
    double sigma;     // |r64| that scaled the current inner phase (0 before the first)
    int scale_exp;    // the batch's fields carry the exact factor 2^scale_exp (float-float outer loop)
};

// (by the exponent bits: a comparison would be one more FP64 instruction)
__device__ __forceinline__ bool finite1(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool finite2(double2 z) { return finite1(z.x) && finite1(z.y); }
// 1/x for 2^-1020 <= |x| < 2^1020 by the hardware's approximation (about 20 bits) and two Newton
// steps, each of which squares the relative error: what is left is rounding, within 2^-52 of
// 1/x.  On GB300 an FP64 instruction of a warp takes about 70 cycles, whatever its
// lanes do, and an IEEE division 750 to 1500 (measured: 8 dependent divisions 12,400
// cycles, 8 of these reciprocals 3,100); the scalar recurrences below sit on every
// iteration's critical path.
__device__ __forceinline__ double fp64_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = ::fma(r, ::fma(-x, r, 1.0), r);
    return ::fma(r, ::fma(-x, r, 1.0), r);
}
// The approximation takes a subnormal for zero and makes a subnormal result zero: outside
// fp64_rcp's range, and for zeros, infinities and NaN, the quotients below divide.
__device__ __forceinline__ bool rcp_in_range(double x) {
    return (unsigned)(((__double2hiint(x) >> 20) & 0x7ff) - 3) < 2040u;  // biased exponent 3 .. 2042
}
__device__ __forceinline__ double fp64_div(double a, double b) { return rcp_in_range(b) ? a * fp64_rcp(b) : a / b; }
__device__ __forceinline__ double2 fp64_div(double2 a, double b) {
    if (!rcp_in_range(b)) return make_double2(a.x / b, a.y / b);
    const double i = fp64_rcp(b);
    return make_double2(a.x * i, a.y * i);
}
// a / b for b2 = |b|^2
__device__ __forceinline__ double2 cdiv_by(double2 a, double2 b, double b2) {
    return fp64_div(make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y), b2);
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) { return cdiv_by(a, b, b.x * b.x + b.y * b.y); }
__device__ __forceinline__ double2 cmul2(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Sum the NV values partials[b][rhs][0 .. NV) over blocks b for one right-hand
// side, by the whole thread block (kScalarThreads threads), in a fixed order:
// strided per-thread sums, lanes, warps.  out[] is valid in thread 0 only.
// FP64 additions are what this costs (a warp's takes 17 to 70 cycles): the
// lanes exchange halves of their 2 NV values instead of each reducing all of
// them (12 additions a warp for NV = 5 instead of 50), warps without a block
// to read drop out, and one lane per value adds the warps.  With the divisions
// of the scalar steps this took scalar_omega_kernel from 14.3 to 4.5 us
// on 64 blocks.
template <int NV>
__device__ __forceinline__ void sum_partials(const double2 *partials, int nblocks, int N, int rhs, double2 (&out)[NV]) {
    constexpr int W = 2 * NV;
    __shared__ double wsum[32][W];
    const int lane = threadIdx.x & 31, nw = min((int)blockDim.x, (nblocks + 31) & ~31) >> 5;
    __syncthreads();  // an earlier call may still be reading wsum
    if ((int)(threadIdx.x >> 5) < nw) {
        double v[W];
#pragma unroll
        for (int k = 0; k < W; ++k) v[k] = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
            const double2 *p = partials + ((size_t)b * N + rhs) * NV;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double2 q = p[k];
                v[2 * k] += q.x;
                v[2 * k + 1] += q.y;
            }
        }
        int idx = 0, end = W, n = W;  // this lane still holds values idx .. end - 1, in v[0 .. n)
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            const int h = (n + 1) / 2;  // (compile-time after unrolling)
            if (n > 1) {
                const bool up = (lane & off) != 0;  // keeps the upper part
#pragma unroll
                for (int k = 0; k < W / 2 + 1; ++k) {
                    if (k >= h) break;
                    const double lo = v[k], hi = h + k < n ? v[h + k] : 0.0;
                    v[k] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, off);
                }
                if (up) idx += h;
                else end = min(end, idx + h);
                n = h;
            } else {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
            }
        }
        if (idx < end) wsum[threadIdx.x >> 5][idx] = v[0];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = 0.0;
        if (lane < W)
            for (int w = 0; w < nw; ++w) t += wsum[w][lane];
#pragma unroll
        for (int k = 0; k < NV; ++k)
            out[k] = make_double2(__shfl_sync(0xffffffffu, t, 2 * k), __shfl_sync(0xffffffffu, t, 2 * k + 1));
    }
}

// Threads per block of the per-right-hand-side scalar kernels (grid = N blocks).
constexpr int kScalarThreads = 256;

// Relative reduction the inner phase aims for: delta, or less when less suffices
// for the outer test |r| <= 0.5 tol min(|bhat|, |b|) (outer_update_kernel), with
// a further factor of 2 for the drift of the low-precision recursive residual.
__device__ __forceinline__ double inner_reduction(const OuterState &o, double delta) {
    if (!(o.r2 > 0.0)) return delta;
    const double need = 0.25 * sqrt(o.tol2 * fmin(o.b2, o.full_b2) / o.r2);
    return fmax(delta, need);
}

// ---------------------------------------------------------------------------
// Scalar recurrences of one right-hand side, shared by the scalar kernels below
// and the cluster-resident solver (resident.cuh).
// ---------------------------------------------------------------------------
__device__ __forceinline__ RhsState begin_state(OuterState &o, double r2, double delta, int max_iters, int max_total,
                                                int fixed) {
    o.sigma = o.active ? sqrt(o.r2) : 0.0;
    RhsState s;
    s.omega = make_double2(1.0, 0.0);
    s.beta = make_double2(0.0, 0.0);
    s.r2 = r2;
    s.r2_0 = r2;
    const double red = inner_reduction(o, delta);
    s.target2 = red * red * r2;
    s.iters = 0;
    s.status = ST_OK;
    const int left = max_total - o.iters;
    s.max_iters = fixed ? max_iters : (max_iters < left ? max_iters : left);
    s.fixed = fixed;
    return s;
}
__device__ __forceinline__ RhsState bicg_begin(OuterState &o, double2 rho, double r2, double delta, int max_iters,
                                               int max_total, int fixed) {
    RhsState s = begin_state(o, r2, delta, max_iters, max_total, fixed);
    s.rho = rho;
    s.alpha = make_double2(1.0, 0.0);
    const bool on = o.active && r2 > 0.0 && isfinite(r2) && (rho.x != 0.0 || rho.y != 0.0) && s.max_iters > 0;
    s.active = on;
    s.next_active = on;
    return s;
}
__device__ __forceinline__ RhsState cg_begin(OuterState &o, double zz, double r2, double delta, int max_iters,
                                             int max_total, int fixed) {
    RhsState s = begin_state(o, r2, delta, max_iters, max_total, fixed);
    s.rho = make_double2(zz, 0.0);
    s.alpha = make_double2(0.0, 0.0);
    s.omega = make_double2(0.0, 0.0);
    const bool on = o.active && r2 > 0.0 && isfinite(r2) && zz > 0.0 && isfinite(zz) && s.max_iters > 0;
    s.active = on;
    s.next_active = on;
    return s;
}
__device__ __forceinline__ void bicg_alpha(RhsState &s, double2 d) {
    s.active = s.next_active;
    if (!s.active) return;
    const double d2 = d.x * d.x + d.y * d.y;
    const double2 a = cdiv_by(s.rho, d, d2);
    if (!(d2 > 0.0) || !finite2(a)) {
        s.status = finite2(d) ? ST_BREAKDOWN : ST_NAN;
        s.active = 0;
        s.next_active = 0;
        return;
    }
    s.alpha = a;
}
__device__ __forceinline__ void bicg_omega(RhsState &s, const double2 (&v)[5]) {
    if (!s.active) return;
    const double2 ts = v[0];
    const double tt = v[1].x;
    const double2 r0s = v[2], r0t = v[3];
    const double ss = v[4].x;
    s.iters += 1;
    bool stop = false;
    if (!(finite1(tt) && finite1(ss) && finite2(ts) && finite2(r0s) && finite2(r0t))) {
        s.status = ST_NAN;
        s.omega = make_double2(0.0, 0.0);
        s.active = 0;  // the vector update is skipped
        s.next_active = 0;
        return;
    }
    const double2 om = fp64_div(ts, tt);
    if (!(tt > 0.0) || !finite2(om)) {
        // t = 0: s is already the solution's residual (zero) or the iteration broke down
        s.omega = make_double2(0.0, 0.0);
        s.r2 = ss;
        s.beta = make_double2(0.0, 0.0);
        if (ss > s.target2) s.status = ST_BREAKDOWN;
        stop = true;
    } else {
        const double2 rho_new = make_double2(r0s.x - (om.x * r0t.x - om.y * r0t.y),
                                             r0s.y - (om.x * r0t.y + om.y * r0t.x));
        double r2 = ss - (ts.x * om.x + ts.y * om.y);
        if (r2 < 0.0) r2 = 0.0;
        s.omega = om;
        s.r2 = r2;
        // beta = (rho'/rho)(alpha/omega), with one reciprocal where the product's square is in its range
        const double2 den = cmul2(s.rho, om);
        const double den2 = den.x * den.x + den.y * den.y;
        const double2 beta = rcp_in_range(den2) ? cdiv_by(cmul2(rho_new, s.alpha), den, den2)
                                                : cmul2(cdiv(rho_new, s.rho), cdiv(s.alpha, om));
        if (!finite2(beta) || !(rho_new.x * rho_new.x + rho_new.y * rho_new.y > 0.0)) {
            s.beta = make_double2(0.0, 0.0);
            if (r2 > s.target2) s.status = ST_BREAKDOWN;
            stop = true;
        } else {
            s.beta = beta;
        }
        s.rho = rho_new;
    }
    const bool done = s.fixed ? (s.iters >= s.max_iters)
                              : (s.r2 <= s.target2 || s.iters >= s.max_iters);
    s.next_active = !(stop || done);
}
__device__ __forceinline__ void cg_alpha(RhsState &s, double ww) {
    s.active = s.next_active;
    if (!s.active) return;
    const double a = fp64_div(s.rho.x, ww);
    if (!(ww > 0.0) || !finite1(a)) {
        s.status = finite1(ww) ? ST_BREAKDOWN : ST_NAN;
        s.active = 0;
        s.next_active = 0;
        return;
    }
    s.alpha = make_double2(a, 0.0);
}
__device__ __forceinline__ void cg_beta(RhsState &s, double r2, double zz) {
    if (!s.active) return;
    s.iters += 1;
    if (!finite1(r2) || !finite1(zz)) {
        s.status = ST_NAN;
        s.active = 0;  // the p update is skipped
        s.next_active = 0;
        return;
    }
    s.r2 = r2;
    bool stop = false;
    if (!(zz > 0.0)) {
        s.beta = make_double2(0.0, 0.0);
        if (r2 > s.target2) s.status = ST_BREAKDOWN;
        stop = true;
    } else {
        s.beta = make_double2(fp64_div(zz, s.rho.x), 0.0);
        s.rho = make_double2(zz, 0.0);
    }
    const bool done = s.fixed ? (s.iters >= s.max_iters) : (s.r2 <= s.target2 || s.iters >= s.max_iters);
    s.next_active = !(stop || done);
}

// ---------------------------------------------------------------------------
// scalar kernels: grid = N blocks of kScalarThreads (one block per right-hand side)
// ---------------------------------------------------------------------------

// Start an inner phase: rho = <rhat, r_l>, r2 = |r_l|^2 (from the partials of
// inner_init_kernel), target and caps; records the scale sigma = |r64| of the
// phase.  max_iters caps this phase; max_total the iterations over all phases.
static __global__ void inner_start_kernel(RhsState *st, OuterState *os, const double2 *partials,
                                   int nblocks, int N, double delta, int max_iters, int max_total, int fixed) {
    const int r = blockIdx.x;
    double2 v[2];
    sum_partials<2>(partials, nblocks, N, r, v);
    const double2 rho = v[0], n2 = v[1];
    if (threadIdx.x != 0) return;
    st[r] = bicg_begin(os[r], rho, n2.x, delta, max_iters, max_total, fixed);
}

// After v = Mhat p: alpha = rho / <rhat, v>.
static __global__ void scalar_alpha_kernel(RhsState *st, const double2 *partials, int nblocks, int N) {
    const int r = blockIdx.x;
    double2 d_[1];
    sum_partials<1>(partials, nblocks, N, r, d_);
    const double2 d = d_[0];
    if (threadIdx.x != 0) return;
    bicg_alpha(st[r], d);
}

// After t = Mhat s: omega, rho', beta, |r'|^2 and the stopping test.
static __global__ void scalar_omega_kernel(RhsState *st, const double2 *partials, int nblocks, int N) {
    const int r = blockIdx.x;
    double2 v[5];
    sum_partials<5>(partials, nblocks, N, r, v);
    if (threadIdx.x != 0) return;
    bicg_omega(st[r], v);
}

static __global__ void count_active_kernel(const RhsState *st, int N, int *out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int n = 0;
        for (int r = 0; r < N; ++r) n += st[r].next_active;
        *out = n;
    }
}

// ---------------------------------------------------------------------------
// vector kernels (even half field, [Vh][12][N]; thread = (element, RHS group))
// ---------------------------------------------------------------------------
struct VecArgs {
    int n_elem;   // Vh * 12
    int N;        // right-hand sides in the layout
};

// s = r - alpha v.  HBM and L2 (3 streams of 201 MB on 16^3 x 32, FP32, width 32:
// 65 us; with the scalars read and converted from FP64 for every element 95 us,
// the conversions sharing the FP64 units).
template <typename S, int R>
static __global__ void __launch_bounds__(256) axpy_s_kernel(VecArgs a, const RhsState *st, const S *r_, const S *v_, S *s_) {
    typedef typename Real<S>::type T;
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    // a thread keeps its right-hand sides (the grid stride is a multiple of G): their scalars are converted once
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    bool any = false;
    cx<T> al[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const RhsState &q = st[r0 + k];
        any |= (q.active != 0);
        al[k] = mk((T)q.alpha.x, (T)q.alpha.y);
    }
    if (!any) return;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const size_t off = ((size_t)(idx >> lgG) * a.N + r0) * 2;
        cx<T> rv[R], vv[R], sv[R];
        ld_pack<S, R, true>(r_ + off, rv);
        ld_pack<S, R, true>(v_ + off, vv);
#pragma unroll
        for (int k = 0; k < R; ++k) sv[k] = rv[k] - al[k] * vv[k];
        st_pack<S, R>(s_ + off, sv);
    }
}

// x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v)
// (5 reads, 3 writes per element while every right-hand side is active: 180 us on
// 16^3 x 32, FP32, width 32, part of s and t still in L2; 249 us with the scalars
// converted per element)
template <typename S, int R>
static __global__ void __launch_bounds__(256) update_kernel(VecArgs a, const RhsState *st, S *x_, S *r_, S *p_,
                                                    const S *s_, const S *t_, const S *v_) {
    typedef typename Real<S>::type T;
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    bool any = false, all = true;
    bool on[R];
    cx<T> al[R], om[R], be[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const RhsState &q = st[r0 + k];
        on[k] = q.active != 0;
        any |= on[k];
        all &= on[k];
        al[k] = mk((T)q.alpha.x, (T)q.alpha.y);
        om[k] = mk((T)q.omega.x, (T)q.omega.y);
        be[k] = mk((T)q.beta.x, (T)q.beta.y);
    }
    if (!any) return;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const size_t off = ((size_t)(idx >> lgG) * a.N + r0) * 2;
        cx<T> xv[R], pv[R], sv[R], tv[R], vv[R], rv[R];
        ld_pack<S, R, false>(x_ + off, xv);
        ld_pack<S, R, false>(p_ + off, pv);
        ld_pack<S, R, true>(s_ + off, sv);
        ld_pack<S, R, true>(t_ + off, tv);
        ld_pack<S, R, true>(v_ + off, vv);
        // the old residual is only needed to keep the entries of inactive right-hand sides
        if (!all) ld_pack<S, R, false>(r_ + off, rv);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (!on[k]) continue;
            xv[k] = xv[k] + al[k] * pv[k] + om[k] * sv[k];
            rv[k] = sv[k] - om[k] * tv[k];
            pv[k] = rv[k] + be[k] * (pv[k] - om[k] * vv[k]);
        }
        st_pack<S, R>(x_ + off, xv);
        st_pack<S, R>(r_ + off, rv);
        st_pack<S, R>(p_ + off, pv);
    }
}

// Inner-phase set-up from the FP64 residual r64 (one of two modes per
// right-hand side):
//  restart:   r_l = r64/|r64| rounded to S; rhat = p = r_l; x_l = 0.
//  continue:  r_l = r64/|r64|; p *= sigma_prev/|r64| (the search direction of the
//             previous phase, rescaled to the new unit); rhat kept; x_l = 0.
//             This is a reliable update (Sleijpen & van der Vorst 1996): the
//             Krylov recurrence carries on and only the residual is replaced by
//             the true one.
// A right-hand side restarts on the first phase, after a breakdown or NaN, or
// when `restart` is set.  Partials: [0] <rhat, r_l> (rho), [1] |r_l|^2, both
// of the rounded values.  Right-hand sides no longer active in the outer loop
// get zero vectors.
template <typename S, int R>
__global__ void __launch_bounds__(256) inner_init_kernel(VecArgs a, const OuterState *os, const RhsState *st,
                                                        const double *r64, S *x_, S *r_, S *rhat_, S *p_,
                                                        double2 *partials, int restart) {
    typedef typename Real<S>::type T;
    extern __shared__ __align__(128) unsigned char smem[];
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    cx<T> red[R][2];
#pragma unroll
    for (int k = 0; k < R; ++k) red[k][0] = red[k][1] = zero<T>();
    // the scales of this thread's right-hand sides: an FP64 root and division per element
    // made this kernel 3.9 times slower (0.83 against 0.215 ms on 16^3 x 32, width 32)
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    double scale[R];
    T pscale[R];
    bool cont[R];
    bool any_cont = false;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const OuterState &o = os[r0 + k];
        const bool on = o.active && o.r2 > 0.0;
        const double root = sqrt(o.r2);
        scale[k] = on ? 1.0 / root : 0.0;
        cont[k] = on && !restart && o.sigma > 0.0 && st[r0 + k].status == ST_OK;
        pscale[k] = cont[k] ? (T)(o.sigma / root) : (T)0;
        any_cont |= cont[k];
    }
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const size_t off = ((size_t)(idx >> lgG) * a.N + r0) * 2;
        cx<double> src[R];
        ld_pack<double, R, true>(r64 + off, src);
        cx<T> lo[R], zr[R], pv[R], rh[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            lo[k] = mk((T)(src[k].re * scale[k]), (T)(src[k].im * scale[k]));
            zr[k] = zero<T>();
        }
        st_pack<S, R>(r_ + off, lo);
        ld_pack<S, R, false>(r_ + off, lo);  // the rounded value, for a consistent rho
        if (any_cont) {
            ld_pack<S, R, false>(p_ + off, pv);
            ld_pack<S, R, false>(rhat_ + off, rh);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (cont[k]) {
                pv[k] = pscale[k] * pv[k];
            } else {
                pv[k] = lo[k];
                rh[k] = lo[k];
            }
        }
        st_pack<S, R>(p_ + off, pv);
        st_pack<S, R>(rhat_ + off, rh);
        ld_pack<S, R, false>(rhat_ + off, rh);
        st_pack<S, R>(x_ + off, zr);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            cjmac(red[k][0], rh[k], lo[k]);
            cjmac(red[k][1], lo[k], lo[k]);
        }
    }
    block_reduce<R, 2, T>(red, G, a.N, partials, smem);
}

// ---------------------------------------------------------------------------
// CG on the normal equations (CGNR: Hestenes-Stiefel CG applied to
// Mhat^dag Mhat e = Mhat^dag r_l), the single-precision solver Sec. 2 uses for
// the low-precision inversions of the truncated solver method.  Mhat is
// gamma5-hermitian (g5 Mhat g5 = Mhat^dag), so Mhat^dag costs the same two
// hops as Mhat.  Per right-hand side and iteration:
//
//   w = Mhat p                       (two hops; |w|^2 fused in the second)
//   alpha = |z|^2 / |w|^2
//   x += alpha p ;  r -= alpha w     (r stored as g5 r; |r|^2 fused)
//   u = Mhat (g5 r)                  (two hops; |u|^2 fused), z' = g5 u = Mhat^dag r
//   beta = |z'|^2 / |z|^2 ;  p = g5 u + beta p
//
// r is the residual of Mhat e = r_l itself, so the inner stopping test
// |r| <= delta |r_l| is the one BiCGStab uses.  RhsState.rho.x holds |z|^2.
// ---------------------------------------------------------------------------

// gamma5 = diag(1, 1, -1, -1) in spin: components 6..11 of a site are negated.
__device__ __forceinline__ bool g5_negates(int e) { return (e % 12) >= 6; }

// Phase set-up: g5 r_l with r_l = r64/|r64| rounded to S; x_l = 0.
// Partials [0] = |r_l|^2 of the rounded value.  Right-hand sides no longer
// active in the outer loop get zero vectors.
template <typename S, int R>
__global__ void __launch_bounds__(256) cg_init_kernel(VecArgs a, const OuterState *os, const double *r64, S *x_,
                                                     S *r5_, double2 *partials) {
    typedef typename Real<S>::type T;
    extern __shared__ __align__(128) unsigned char smem[];
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    cx<T> red[R][1];
#pragma unroll
    for (int k = 0; k < R; ++k) red[k][0] = zero<T>();
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    double scale[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const OuterState &o = os[r0 + k];
        scale[k] = (o.active && o.r2 > 0.0) ? 1.0 / sqrt(o.r2) : 0.0;
    }
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int e = (int)(idx >> lgG);
        const size_t off = ((size_t)e * a.N + r0) * 2;
        const bool neg = g5_negates(e);
        cx<double> src[R];
        ld_pack<double, R, true>(r64 + off, src);
        cx<T> lo[R], zr[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const double sc = neg ? -scale[k] : scale[k];
            lo[k] = mk((T)(src[k].re * sc), (T)(src[k].im * sc));
            zr[k] = zero<T>();
        }
        st_pack<S, R>(r5_ + off, lo);
        ld_pack<S, R, false>(r5_ + off, lo);  // the rounded value
        st_pack<S, R>(x_ + off, zr);
#pragma unroll
        for (int k = 0; k < R; ++k) cjmac(red[k][0], lo[k], lo[k]);
    }
    block_reduce<R, 1, T>(red, G, a.N, partials, smem);
}

// x += alpha p ;  g5 r -= alpha g5 w  for active right-hand sides; partials [0] = |r|^2.
template <typename S, int R>
__global__ void __launch_bounds__(256) cg_update_kernel(VecArgs a, const RhsState *st, S *x_, S *r5_, const S *p_,
                                                       const S *w_, double2 *partials) {
    typedef typename Real<S>::type T;
    extern __shared__ __align__(128) unsigned char smem[];
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    cx<T> red[R][1];
#pragma unroll
    for (int k = 0; k < R; ++k) red[k][0] = zero<T>();
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    bool on[R];
    bool any = false;
    T al[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const RhsState &q = st[r0 + k];
        on[k] = q.active != 0;
        any |= on[k];
        al[k] = (T)q.alpha.x;
    }
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; any && idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int e = (int)(idx >> lgG);
        const T sg = g5_negates(e) ? (T)-1 : (T)1;
        const size_t off = ((size_t)e * a.N + r0) * 2;
        cx<T> xv[R], rv[R], pv[R], wv[R];
        ld_pack<S, R, false>(x_ + off, xv);
        ld_pack<S, R, false>(r5_ + off, rv);
        ld_pack<S, R, true>(p_ + off, pv);
        ld_pack<S, R, true>(w_ + off, wv);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (!on[k]) continue;
            xv[k] = xv[k] + al[k] * pv[k];
            rv[k] = rv[k] - (sg * al[k]) * wv[k];
        }
        st_pack<S, R>(x_ + off, xv);
        st_pack<S, R>(r5_ + off, rv);
        ld_pack<S, R, false>(r5_ + off, rv);  // the rounded value
#pragma unroll
        for (int k = 0; k < R; ++k) cjmac(red[k][0], rv[k], rv[k]);
    }
    block_reduce<R, 1, T>(red, G, a.N, partials, smem);
}

// p = g5 u + beta p for active right-hand sides, or p = g5 u everywhere (init).
template <typename S, int R>
__global__ void __launch_bounds__(256) cg_p_kernel(VecArgs a, const RhsState *st, const S *u_, S *p_, int init) {
    typedef typename Real<S>::type T;
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    bool on[R];
    bool any = false;
    T be[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const RhsState &q = st[r0 + k];
        on[k] = init || q.active != 0;
        any |= on[k];
        be[k] = init ? (T)0 : (T)q.beta.x;
    }
    if (!any) return;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int e = (int)(idx >> lgG);
        const T sg = g5_negates(e) ? (T)-1 : (T)1;
        const size_t off = ((size_t)e * a.N + r0) * 2;
        cx<T> uv[R], pv[R];
        ld_pack<S, R, true>(u_ + off, uv);
        if (init) {
#pragma unroll
            for (int k = 0; k < R; ++k) pv[k] = sg * uv[k];
        } else {
            ld_pack<S, R, false>(p_ + off, pv);
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (on[k]) pv[k] = sg * uv[k] + be[k] * pv[k];
        }
        st_pack<S, R>(p_ + off, pv);
    }
}

// CG phase start: |r_l|^2 from cg_init_kernel's partials (pr), |z|^2 = |u|^2
// from the second hop of u = Mhat g5 r_l (pu); target, caps and sigma as in
// inner_start_kernel.
static __global__ void cg_start_kernel(RhsState *st, OuterState *os, const double2 *pr, int nr, const double2 *pu,
                                       int nu, int N, double delta, int max_iters, int max_total, int fixed) {
    const int r = blockIdx.x;
    double2 n2_[1];
    sum_partials<1>(pr, nr, N, r, n2_);
    const double2 n2 = n2_[0];
    double2 zz_[1];
    sum_partials<1>(pu, nu, N, r, zz_);
    const double2 zz = zz_[0];
    if (threadIdx.x != 0) return;
    st[r] = cg_begin(os[r], zz.x, n2.x, delta, max_iters, max_total, fixed);
}

// After w = Mhat p: alpha = |z|^2 / |w|^2.
static __global__ void cg_alpha_kernel(RhsState *st, const double2 *partials, int nblocks, int N) {
    const int r = blockIdx.x;
    double2 ww_[1];
    sum_partials<1>(partials, nblocks, N, r, ww_);
    const double2 ww = ww_[0];
    if (threadIdx.x != 0) return;
    cg_alpha(st[r], ww.x);
}

// After the update (pr: |r|^2) and u = Mhat g5 r (pu: |u|^2): beta, stopping test.
static __global__ void cg_beta_kernel(RhsState *st, const double2 *pr, int nr, const double2 *pu, int nu, int N) {
    const int r = blockIdx.x;
    double2 n2_[1];
    sum_partials<1>(pr, nr, N, r, n2_);
    const double2 n2 = n2_[0];
    double2 zz_[1];
    sum_partials<1>(pu, nu, N, r, zz_);
    const double2 zz = zz_[0];
    if (threadIdx.x != 0) return;
    cg_beta(st[r], n2.x, zz.x);
}

// x64 += |r64| * x_l for right-hand sides active in the outer loop.
template <typename S, int R>
static __global__ void __launch_bounds__(256) accumulate_kernel(VecArgs a, const OuterState *os, const S *x_, double *x64) {
    typedef typename Real<S>::type T;
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    const int r0 = (int)(threadIdx.x & (G - 1)) * R;
    double sc[R];
    bool on[R], any = false;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        on[k] = os[r0 + k].active != 0;
        any |= on[k];
        sc[k] = on[k] ? sqrt(os[r0 + k].r2) : 0.0;
    }
    if (!any) return;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const size_t off = ((size_t)(idx >> lgG) * a.N + r0) * 2;
        cx<T> xl[R];
        ld_pack<S, R, true>(x_ + off, xl);
        cx<double> acc[R];
        ld_pack<double, R, false>(x64 + off, acc);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (on[k]) {
                acc[k].re += sc[k] * (double)xl[k].re;
                acc[k].im += sc[k] * (double)xl[k].im;
            }
        }
        st_pack<double, R>(x64 + off, acc);
    }
}

// ---------------------------------------------------------------------------
// outer (FP64) bookkeeping: grid = N blocks of kScalarThreads
// ---------------------------------------------------------------------------
// mode 0: initialise (b2 = |bhat|^2 from partials, r2 = b2, active = b2 > 0)
// mode 1: after the true residual r (partials: |r|^2, which is also the
//         full-lattice residual): r2, full_r2, convergence test, cycle count
// mode 2: after a fixed-iteration phase and its residual: full_r2 and the
//         cycle and iteration counts only
static __global__ void outer_update_kernel(OuterState *os, const RhsState *st, const double2 *partials, int nblocks,
                                    int N, int mode, double tol, int max_outer, int max_iter) {
    const int r = blockIdx.x;
    double2 n2_[1];
    sum_partials<1>(partials, nblocks, N, r, n2_);
    const double2 n2 = n2_[0];
    if (threadIdx.x != 0) return;
    OuterState &o = os[r];
    if (mode == 0) {
        o.b2 = n2.x;
        o.r2 = n2.x;
        o.tol2 = tol * tol;
        o.outer = 0;
        o.iters = 0;
        o.sigma = 0.0;
        o.status = ST_OK;
        o.active = (n2.x > 0.0) ? 1 : 0;
        if (!isfinite(n2.x)) { o.status = ST_NAN; o.active = 0; }
        return;
    }
    o.full_r2 = n2.x;  // every right-hand side: an inactive one's x is unchanged
    if (!o.active) return;
    o.outer += 1;
    o.iters += st[r].iters;
    if (st[r].status == ST_NAN) o.status = ST_NAN;
    if (mode == 2) return;
    o.r2 = n2.x;
    if (!isfinite(n2.x)) {
        o.status = ST_NAN;
        o.active = 0;
    } else if (n2.x <= 0.25 * o.tol2 * fmin(o.b2, o.full_b2)) {
        // half the tolerance on the Schur system, measured against the smaller of
        // |bhat| and |b|, so that the full-lattice residual |b - M x|/|b| meets tol
        o.active = 0;
    } else if (o.outer >= max_outer || o.iters >= max_iter) {
        o.active = 0;  // reported as not converged by the host
    }
}

static __global__ void outer_count_kernel(const OuterState *os, int N, int *out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int n = 0;
        for (int r = 0; r < N; ++r) n += os[r].active;
        *out = n;
    }
}

// Exact power-of-two scale of each right-hand side for the float-float outer
// loop, whose numbers keep only the float exponent range (about 1e-38 to 3e38,
// and their low words lose bits below about 1e-31 of that range): k_r =
// -ilogb(|b_r|), so the scaled source has a norm in [1, 2).  A zero or
// non-finite norm keeps k_r = 0.  One thread per right-hand side.
static __global__ void pow2_pick_kernel(OuterState *os, int N) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= N) return;
    const double b2 = os[r].full_b2;
    os[r].scale_exp = (b2 > 0.0 && isfinite(b2)) ? -ilogb(sqrt(b2)) : 0;
}

// 2^e as a double for e in [-1022, 1023] (built from its bits, exact).
__device__ __forceinline__ double pow2_exact(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// f[e][r] *= 2^(sign * k_r) on a field of n_rows rows of N complex doubles (N a
// power of two dividing the block size, so a thread always meets the same
// right-hand side r = index mod N).  2^k is applied as two factors 2^(k/2) and
// 2^(k - k/2), each a normal double for |k| <= 2046; the products are exact
// unless a value under- or overflows.
static __global__ void pow2_scale_kernel(double *f, size_t n_rows, int N, const OuterState *os, int sign) {
    const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const int k = sign * os[first & (size_t)(N - 1)].scale_exp;
    if (k == 0) return;
    const double f1 = pow2_exact(k / 2), f2 = pow2_exact(k - k / 2);
    double2 *z = reinterpret_cast<double2 *>(f);
    const size_t total = n_rows * (size_t)N;
    for (size_t i = first; i < total; i += stride) {
        double2 v = z[i];
        v.x = v.x * f1 * f2;
        v.y = v.y * f1 * f2;
        z[i] = v;
    }
}

// full-system norms: mode 0 -> full_b2 (sum of two partial sets), mode 1 -> full_r2
static __global__ void full_norm_kernel(OuterState *os, const double2 *pa, int na, const double2 *pb, int nb, int N,
                                 int mode) {
    const int r = blockIdx.x;
    double2 a_[1];
    sum_partials<1>(pa, na, N, r, a_);
    const double2 a = a_[0];
    double2 b_[1];
    sum_partials<1>(pb, nb, N, r, b_);
    const double2 b = b_[0];
    if (threadIdx.x != 0) return;
    if (mode == 0) os[r].full_b2 = a.x + b.x;
    else os[r].full_r2 = a.x + b.x;
}

}  // namespace dl

namespace dl {
// |v|^2 per right-hand side of a half field -> partials
template <typename S, int R>
static __global__ void __launch_bounds__(256) norm2_kernel(VecArgs a, const S *v_, double2 *partials) {
    typedef typename Real<S>::type T;
    extern __shared__ __align__(128) unsigned char smem[];
    const int G = a.N / R, lgG = __ffs(G) - 1;
    const long total = (long)a.n_elem << lgG;  // elements x groups: may exceed 2^31
    cx<T> red[R][1];
#pragma unroll
    for (int k = 0; k < R; ++k) red[k][0] = zero<T>();
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int e = (int)(idx >> lgG), r0 = (int)(idx & (G - 1)) * R;
        cx<T> v[R];
        ld_pack<S, R, true>(v_ + ((size_t)e * a.N + r0) * 2, v);
#pragma unroll
        for (int k = 0; k < R; ++k)  // (the imaginary part of <v, v> is not read)
            red[k][0].re = ::fma(v[k].re, v[k].re, ::fma(v[k].im, v[k].im, red[k][0].re));
    }
    block_reduce<R, 1, T>(red, G, a.N, partials, smem);
}

// FP64 <-> storage type S over n_complex values: to_lo = 1 rounds FP64 to S the
// way the solver's inner phase does (to float, then to S), to_lo = 0 widens S to
// FP64 exactly.
template <typename S>
static __global__ void cast_kernel(double *f64, S *lo, size_t n_complex, int to_lo) {
    typedef typename Real<S>::type T;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_complex; i += (size_t)gridDim.x * blockDim.x) {
        if (to_lo) {
            const double2 v = reinterpret_cast<const double2 *>(f64)[i];
            cx<T> z[1] = {mk((T)v.x, (T)v.y)};
            st_pack<S, 1>(lo + 2 * i, z);
        } else {
            cx<T> z[1];
            ld_pack<S, 1, false>(lo + 2 * i, z);
            reinterpret_cast<double2 *>(f64)[i] = make_double2((double)z[0].re, (double)z[0].im);
        }
    }
}

// deterministic pseudo-random fill (for timing runs only)
template <typename S>
static __global__ void fill_kernel(S *v, size_t n_complex, uint32_t seed) {
    typedef typename Real<S>::type T;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_complex; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t h = (uint32_t)i * 2654435761u ^ seed;
        h ^= h >> 15; h *= 2246822519u; h ^= h >> 13;
        cx<T> z[1];
        z[0] = mk((T)((h & 0xffff) / 65536.0 - 0.5), (T)((h >> 16) / 65536.0 - 0.5));
        st_pack<S, 1>(v + 2 * i, z);
    }
}
}  // namespace dl
