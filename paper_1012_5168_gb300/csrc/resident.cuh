// Cluster-resident Krylov solver: a whole inner phase (BiCGStab or CGNR, FP32 or BF16
// fields) of a mixed-precision solve in one launch, for problems that live in L2.
//
// On a small lattice the step-by-step iteration (eight launches: four hops,
// two vector updates, two scalar kernels) is bound by launch gaps and by the
// latency of nearly empty kernels: one right-hand side on 8^3 x 16 took 53 us
// per iteration for about 4 us of memory traffic.  Here a thread-block cluster
// of C SMs takes one right-hand side and iterates it to the end by itself.  The
// right-hand sides are independent, so clusters never wait for one another: no
// grid-wide barrier and no co-residency requirement, and a cluster retires as
// soon as its right-hand side stops.  Inside a cluster the phases of an
// iteration are separated by the hardware cluster barrier, and the reductions
// travel through distributed shared memory: every block sums all C partials in
// rank order and repeats the scalar recurrences, so all blocks take the same
// decisions without a further exchange.  (Several right-hand sides per cluster
// share the links, but with the same SMs each cluster then needs more blocks:
// on 8^3 x 16 with 32 right-hand sides 1 x 4 blocks ran at 8.5 ms a solve, 2 x 8
// at 14, 4 x 16 at 15.)
//
// Latency.  With one thread per site the eight directions of a hop became
// eight load round trips (7500 cycles for a hop of 128 sites).  So four warps
// share 32 sites, warp q taking direction mu = q forward and backward: all 33
// loads of a thread are in flight at once, the four partial sums meet in shared
// memory, and warp q goes on with spin q (three of the twelve components) in
// the epilogue and in the vector updates (3400 cycles).  The vector updates load two
// sites a step, and the coordinates are computed (every cluster barrier empties L1 of a
// table of them): CGNR on 8^3 x 16 from 11.0 to 10.2 ms a solve (12.2 ms step by step), 24
// right-hand sides of a fermion force there from 24.5 to 22.3 ms (30.0 ms).
//
// Layout.  The inner fields belong to this kernel alone: per right-hand side
// [tile of 32 sites][12][32] complex.  A warp reads 256 contiguous bytes per
// component, where the layout of the other kernels would touch 32 lines per
// load for a single right-hand side; the component offsets are immediates, and
// no power-of-two stride separates the components.  Links are [parity][tile of
// 32 sites][36][32] pairs of consecutive elements of the eight-link row
// (time-boundary factor folded in): one 16-byte load per lane gives two FP32
// link elements.  Block k of a cluster owns a contiguous range of sites of both
// parities, so most x, y and z neighbours of its sites are its own.
//
// The recurrences are those of blas.cuh, rounded at the same places (fields in
// storage type S, arithmetic in Real<S>, scalars in FP64); only the order of
// the reduction sums differs.
#pragma once

#include <cooperative_groups.h>

#include "blas.cuh"
#include "hop.cuh"

namespace dl {

constexpr int RES_THREADS = 512;               // one block per SM, 128 registers a thread
constexpr int RES_GROUPS = RES_THREADS / 128;  // groups of four warps, 32 sites each
constexpr int RES_ROUND = 32 * RES_GROUPS;     // sites of a block in flight
constexpr int RES_MAX_C = 16;                  // blocks per cluster

// Complex values of one right-hand side's inner field, and of the links of both parities.
inline size_t res_field_elems(long Vh) { return (size_t)((Vh + 31) / 32) * 384; }
inline size_t res_link_elems(long Vh) { return (size_t)2 * ((Vh + 31) / 32) * 32 * 72; }

struct ResArgs {
    void *f[8];             // x r rhat p v s t tmp: [rhs][tile][12][32] complex of S
    const void *links;      // [2][tile][36][32] pairs of complex of S
    Geom g;
    uint32_t div[3];        // floor(2^32 / d) + 1 for d = L_x, L_y, L_z
    int N;                  // width of the FP64 fields
    double k2;              // kappa^2
    RhsState *st;
    OuterState *os;
    const double *src;      // FP64 residual, even half [Vh][12][N]
    double *x64;            // even half of the solution, += |r64| x_l
    double delta;
    int max_iters, max_total, fixed;
};

template <typename S> __device__ __forceinline__ cx<typename Real<S>::type> res_round(cx<typename Real<S>::type> z) {
    uint32_t w[Conv<S>::W];
    Conv<S>::put(z, w);
    return Conv<S>::get(w);
}

// Component c of the site at tile offset t (complex units, component 0).
template <typename S> __device__ __forceinline__ cx<typename Real<S>::type> res_ld(const S *f, uint32_t t, int c) {
    cx<typename Real<S>::type> v[1];
    ld_pack<S, 1, false>(f + 2 * ((size_t)t + c * 32), v);
    return v[0];
}
template <typename S> __device__ __forceinline__ void res_st(S *f, uint32_t t, int c, cx<typename Real<S>::type> z) {
    cx<typename Real<S>::type> v[1] = {z};
    st_pack<S, 1>(f + 2 * ((size_t)t + c * 32), v);
}
__device__ __forceinline__ uint32_t res_tile(uint32_t e) { return (e >> 5) * 384 + (e & 31); }

template <typename T>
struct ResShared {
    cx<T> part[RES_GROUPS][4][9][32];                // partial hop sums: [group][mu][other spins][site]
    double2 slot[2][RES_MAX_C][5];                   // [buffer][rank]: every block's partial sums
    cx<T> warp[RES_THREADS / 32][5];                 // partial sums of the warps
    double2 total[5];
    RhsState rhs;
    cx<T> alpha, omega, beta;                        // the scalars in arithmetic precision
    int active, next;
};
// A conversion from FP64 costs about as much as an FP64 instruction: one thread
// makes them for all.
template <typename T> __device__ __forceinline__ void res_publish(ResShared<T> &sh) {
    const RhsState &s = sh.rhs;
    sh.alpha = mk((T)s.alpha.x, (T)s.alpha.y);
    sh.omega = mk((T)s.omega.x, (T)s.omega.y);
    sh.beta = mk((T)s.beta.x, (T)s.beta.y);
    sh.active = s.active;
    sh.next = s.next_active;
}

// Coordinates of checkerboard site cb of parity par: quotients n / d by multiplication, exact
// for n d < 2^32 and d > 1 (n is below 2^15 here, an extent at most 256).  A table of them would be one more load
// round trip, since every cluster barrier empties L1.
__device__ __forceinline__ Site res_site(int cb, int par, const Geom &g, const uint32_t (&div)[3]) {
    Site s;
    const int row = (int)__umulhi(2 * (uint32_t)cb, div[0]), zt = (int)__umulhi((uint32_t)row, div[1]);
    const int t = (int)__umulhi((uint32_t)zt, div[2]);
    s.c[1] = row - zt * g.L[1];
    s.c[2] = zt - t * g.L[2];
    s.c[3] = t;
    s.c[0] = 2 * (cb - row * (g.L[0] >> 1)) + ((s.c[1] + s.c[2] + t + par) & 1);
    s.i = 2 * cb + (s.c[0] & 1);
    return s;
}

// Barrier of the four warps of a group.
__device__ __forceinline__ void res_bar(int grp) { asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory"); }

// The NV complex sums over the cluster of the threads' red[], into sh.total of
// every block, in a fixed order: lanes, warps (four runs), ranks (four runs).
// Contains the cluster barrier that also orders the phase's field stores.  With C > 1 it
// writes into the other blocks' shared memory: a cluster barrier must lie before the first call.
template <int NV, typename T>
__device__ __forceinline__ void res_sum(ResShared<T> &sh, cx<T> (&red)[NV], int C, int rank, int buf) {
    const int tid = threadIdx.x, lane = tid & 31;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            red[k].re += shfl_xor(red[k].re, off);
            red[k].im += shfl_xor(red[k].im, off);
        }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh.warp[tid >> 5][k] = red[k];
    __syncthreads();
    // four lanes per real value
    const int q = tid & 3, o = tid >> 2;
    constexpr int per = RES_THREADS / 128;  // warps per lane
    if (tid < ((2 * NV * 4 + 31) & ~31)) {
        double v = 0.0;
        if (o < 2 * NV) {
            const T *w = reinterpret_cast<const T *>(sh.warp[q * per]) + o;
#pragma unroll
            for (int k = 0; k < per; ++k) v += (double)w[k * 10];
        }
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (o < 2 * NV) {
            if (C == 1) {
                if (q == 0) reinterpret_cast<double *>(sh.total)[o] = v;
            } else {
                auto cl = cooperative_groups::this_cluster();
                double *slot = reinterpret_cast<double *>(sh.slot[buf][rank]);
                for (int k = q; k < C; k += 4) cl.map_shared_rank(slot, k)[o] = v;
            }
        }
    }
    if (C == 1) {
        __syncthreads();
        return;
    }
    cooperative_groups::this_cluster().sync();
    if (tid < ((2 * NV * 4 + 31) & ~31)) {
        double v = 0.0;
        if (o < 2 * NV)
            for (int k = q * C / 4; k < (q + 1) * C / 4; ++k) v += reinterpret_cast<const double *>(sh.slot[buf][k])[o];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (o < 2 * NV && q == 0) reinterpret_cast<double *>(sh.total)[o] = v;
    }
    __syncthreads();
}

// The direction pair mu of the hop of one item: its contribution to spin MU in
// own[], to the other spins in part[][lane].
template <typename S, int MU>
__device__ __forceinline__ void res_mu(const S *in, const S *lk, const Geom &g, const Site &st,
                                       cx<typename Real<S>::type> (&own)[3],
                                       cx<typename Real<S>::type> (*part)[32], int lane) {
    typedef typename Real<S>::type T;
    cx<T> u[9], v[9], hf[1][6], hb[1][6], w[6], acc[12];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        cx<T> two[2];
        ld_pack<S, 2, true>(lk + (9 * MU + k) * 128, two);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (2 * k + h < 9) u[2 * k + h] = two[h];
            else v[2 * k + h - 9] = two[h];
        }
    }
    const uint32_t tf = res_tile(nbr_fwd(st, g, MU)), tb = res_tile(nbr_bwd(st, g, MU));
    load_project<S, 1, MU, -1, false>(in + 2 * (size_t)tf, 32, hf);
    load_project<S, 1, MU, +1, false>(in + 2 * (size_t)tb, 32, hb);
    // w+ = U h+ and w- = V^dag h-: the pair contributes [w+ + w-; X^dag (w- - w+)], X being the
    // projection's map (no sums with zeros, and one permutation for both)
    su3_mul<T, false>(u, hf[0], w);
    {
        cx<T> y[6];
        su3_mul<T, true>(v, hb[0], y);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            acc[k] = w[k] + y[k];
            w[k] = y[k] - w[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        acc[6 + k] = MU == 0 ? tmi(w[3 + k]) : MU == 1 ? w[3 + k] : MU == 2 ? tmi(w[k]) : w[k];
        acc[9 + k] = MU == 0 ? tmi(w[k]) : MU == 1 ? -w[k] : MU == 2 ? ti(w[3 + k]) : w[3 + k];
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (s == MU) own[a] = acc[3 * s + a];
            else part[(s - (s > MU ? 1 : 0)) * 3 + a][lane] = acc[3 * s + a];
        }
}

template <typename S, int CG>
__global__ void __launch_bounds__(RES_THREADS, 1) resident_kernel(ResArgs A) {
    typedef typename Real<S>::type T;
    extern __shared__ __align__(128) unsigned char smem[];
    ResShared<T> &sh = *reinterpret_cast<ResShared<T> *>(smem);
    auto cluster = cooperative_groups::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int rg = blockIdx.x / C;  // the right-hand side
    const int tid = threadIdx.x, lane = tid & 31, q = (tid >> 5) & 3, grp = tid >> 7;
    const int Vh = A.g.Vh;
    // this block's sites: whole tiles where there are enough of them
    const int unit = Vh >= 256 * C ? 32 : 1, nu = (Vh + unit - 1) / unit;
    const int c0 = min(Vh, (int)((long)nu * rank / C) * unit), c1 = min(Vh, (int)((long)nu * (rank + 1) / C) * unit);
    const int nit = c1 - c0;
    const size_t gb = (size_t)rg * ((Vh + 31) / 32) * 768;
    S *X = (S *)A.f[0] + gb, *R = (S *)A.f[1] + gb, *RH = (S *)A.f[2] + gb, *P = (S *)A.f[3] + gb;
    S *V = (S *)A.f[4] + gb, *SS = (S *)A.f[5] + gb, *TT = (S *)A.f[6] + gb, *TMP = (S *)A.f[7] + gb;
    const T mk2 = (T)-A.k2;
    const int first = grp * 32 + lane;  // this thread's first site; the next ones are RES_ROUND apart
    const int c3 = 3 * q;               // its components c3 .. c3 + 2 (spin q)

    auto fence = [&] {
        if (C == 1) __syncthreads();
        else cluster.sync();
    };
    // spin q of D in at site i of parity `par`; every lane of the
    // group's four warps calls it, those with i >= n without a site
    auto hop = [&](const S *in, int par, int i, int n, cx<T>(&d)[3]) {
        const int cb = c0 + i;
        cx<T>(*part)[32] = sh.part[grp][q];
        if (i < n) {
            const Site st = res_site(cb, par, A.g, A.div);
            const S *lk = (const S *)A.links +
                          ((size_t)(par * ((Vh + 31) >> 5) + (cb >> 5)) * 36 * 32 + (cb & 31)) * 4;
            if (q == 0) res_mu<S, 0>(in, lk, A.g, st, d, part, lane);
            else if (q == 1) res_mu<S, 1>(in, lk, A.g, st, d, part, lane);
            else if (q == 2) res_mu<S, 2>(in, lk, A.g, st, d, part, lane);
            else res_mu<S, 3>(in, lk, A.g, st, d, part, lane);
        }
        res_bar(grp);
#pragma unroll
        for (int m = 1; m < 4; ++m) {  // the other directions in cyclic order
            const int mu = (q + m) & 3, row = (q - (q > mu ? 1 : 0)) * 3;
#pragma unroll
            for (int a = 0; a < 3; ++a) d[a] = d[a] + sh.part[grp][mu][row + a][lane];
        }
        res_bar(grp);
    };

    // A block's shared memory may be written from another block only once it has started, and
    // the set-up's res_sum is the first to do so.
    if (C > 1) cluster.sync();

    // ---- phase set-up: fields from the FP64 residual
    const OuterState &o = A.os[rg];
    const double sc0 = o.active && o.r2 > 0.0 ? 1.0 / sqrt(o.r2) : 0.0;
    {
        cx<T> red[2] = {zero<T>(), zero<T>()};
        for (int i = first; i < nit; i += RES_ROUND) {
            const int cb = c0 + i;
            const uint32_t t = res_tile(c0 + i);
            const double sc = (CG && q >= 2) ? -sc0 : sc0;  // CG keeps g5 r
            double2 v[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                v[a] = __ldg(reinterpret_cast<const double2 *>(A.src) + ((size_t)cb * 12 + c3 + a) * A.N + rg);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const cx<T> lo = res_round<S>(mk((T)(v[a].x * sc), (T)(v[a].y * sc)));
                res_st<S>(R, t, c3 + a, lo);
                res_st<S>(X, t, c3 + a, zero<T>());
                if (!CG) {
                    res_st<S>(RH, t, c3 + a, lo);
                    res_st<S>(P, t, c3 + a, lo);
                }
                cjmac(red[0], lo, lo);
            }
        }
        if (CG) {  // u = Mhat g5 r, p = g5 u: its norm starts the recurrence
            fence();
            for (int i = first; (i & ~31) < nit; i += RES_ROUND) {
                cx<T> d[3];
                hop(R, 1, i, nit, d);
                if (i < nit)
#pragma unroll
                    for (int a = 0; a < 3; ++a) res_st<S>(TMP, res_tile(c0 + i), c3 + a, d[a]);
            }
            fence();
            for (int i = first; (i & ~31) < nit; i += RES_ROUND) {
                cx<T> d[3];
                hop(TMP, 0, i, nit, d);
                if (i < nit)
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const uint32_t t = res_tile(c0 + i);
                        const cx<T> u = res_ld<S>(R, t, c3 + a) + mk2 * d[a], ur = res_round<S>(u);
                        res_st<S>(P, t, c3 + a, q >= 2 ? -ur : ur);
                        cjmac(red[1], u, u);
                    }
            }
        }
        res_sum<2>(sh, red, C, rank, 0);
        if (tid == 0) {
            OuterState oo = A.os[rg];
            const double n2 = sh.total[0].x, zz = sh.total[1].x;
            sh.rhs = CG ? cg_begin(oo, zz, n2, A.delta, A.max_iters, A.max_total, A.fixed)
                             : bicg_begin(oo, make_double2(n2, 0.0), n2, A.delta, A.max_iters, A.max_total, A.fixed);
            res_publish(sh);
        }
        __syncthreads();
    }
    // ---- iterations: every right-hand side stops after at most max_iters of them
    for (int it = 0; it < A.max_iters; ++it) {
        if (!sh.next) break;
        cx<T> red[CG ? 2 : 5];
#pragma unroll
        for (int k = 0; k < (CG ? 2 : 5); ++k) red[k] = zero<T>();
        cx<T> al = zero<T>();
        S *const W = CG ? R : SS;  // the field of the second matrix product
        int n = nit;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {  // v = Mhat p, then t = Mhat s (CG: u = Mhat g5 r)
            S *const Y = half ? W : P, *const O = half ? TT : V;
            cx<T> dot = zero<T>();
#pragma unroll 1
            for (int par = 1; par >= 0; --par) {  // one copy of the hop's code serves all four hops
                const S *in = par ? Y : TMP;
#pragma unroll 1
                for (int i = first; (i & ~31) < nit; i += RES_ROUND) {
                    const uint32_t t = res_tile(c0 + i);
                    cx<T> d[3], y[3], rh[3];
                    if (!par && i < n) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            y[a] = res_ld<S>(Y, t, c3 + a);
                            if (!CG) rh[a] = res_ld<S>(RH, t, c3 + a);
                        }
                    }
                    hop(in, par, i, n, d);
                    if (i >= n) continue;
                    if (par) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) res_st<S>(TMP, t, c3 + a, d[a]);
                        continue;
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const cx<T> z = y[a] + mk2 * d[a];
                        res_st<S>(O, t, c3 + a, z);
                        if constexpr (CG != 0) {
                            cjmac(dot, z, z);
                        } else if (half == 0) {
                            cjmac(dot, rh[a], z);
                        } else {
                            cjmac(red[0], z, y[a]);
                            cjmac(red[1], z, z);
                            cjmac(red[2], rh[a], y[a]);
                            cjmac(red[3], rh[a], z);
                            cjmac(red[4], y[a], y[a]);
                        }
                    }
                }
                if (par) fence();
            }
            if (half) {
                if (CG) red[1] = dot;
                break;
            }
            cx<T> one[1] = {dot};
            res_sum<1>(sh, one, C, rank, 0);
            if (tid == 0) {
                if (CG) cg_alpha(sh.rhs, sh.total[0].x);
                else bicg_alpha(sh.rhs, sh.total[0]);
                res_publish(sh);
            }
            __syncthreads();
            n = sh.active ? nit : 0;  // after a breakdown nothing more is touched
            al = sh.alpha;
            for (int i0 = first; i0 < n; i0 += 2 * RES_ROUND) {  // two sites' loads in flight
                cx<T> rv[2][3], vv[2][3], xv[2][3], pv[2][3];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = i0 + h * RES_ROUND;
                    const uint32_t t = res_tile(c0 + (i < n ? i : i0));
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        rv[h][a] = res_ld<S>(R, t, c3 + a);
                        vv[h][a] = res_ld<S>(V, t, c3 + a);
                        if (CG) {
                            xv[h][a] = res_ld<S>(X, t, c3 + a);
                            pv[h][a] = res_ld<S>(P, t, c3 + a);
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = i0 + h * RES_ROUND;
                    if (i >= n) break;
                    const uint32_t t = res_tile(c0 + i);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        if (CG) {
                            res_st<S>(X, t, c3 + a, xv[h][a] + al.re * pv[h][a]);
                            const cx<T> z = res_round<S>(rv[h][a] - (q >= 2 ? -al.re : al.re) * vv[h][a]);
                            res_st<S>(R, t, c3 + a, z);
                            cjmac(red[0], z, z);
                        } else {
                            res_st<S>(SS, t, c3 + a, rv[h][a] - al * vv[h][a]);
                        }
                    }
                }
            }
            fence();
        }
        res_sum(sh, red, C, rank, 1);
        if (tid == 0) {
            if constexpr (CG != 0) {
                cg_beta(sh.rhs, sh.total[0].x, sh.total[1].x);
            } else {
                double2 v[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) v[k] = sh.total[k];
                bicg_omega(sh.rhs, v);
            }
            res_publish(sh);
        }
        __syncthreads();
        const cx<T> om = sh.omega, be = sh.beta;
        n = sh.active ? nit : 0;
        for (int i0 = first; i0 < n; i0 += 2 * RES_ROUND) {
            cx<T> xv[2][3], pv[2][3], sv[2][3], tv[2][3], vv[2][3];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = i0 + h * RES_ROUND;
                const uint32_t t = res_tile(c0 + (i < n ? i : i0));
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    pv[h][a] = res_ld<S>(P, t, c3 + a);
                    tv[h][a] = res_ld<S>(TT, t, c3 + a);
                    if (!CG) {
                        xv[h][a] = res_ld<S>(X, t, c3 + a);
                        sv[h][a] = res_ld<S>(SS, t, c3 + a);
                        vv[h][a] = res_ld<S>(V, t, c3 + a);
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = i0 + h * RES_ROUND;
                if (i >= n) break;
                const uint32_t t = res_tile(c0 + i);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (CG) {
                        res_st<S>(P, t, c3 + a, (q >= 2 ? (T)-1 : (T)1) * tv[h][a] + be.re * pv[h][a]);
                    } else {
                        res_st<S>(X, t, c3 + a, xv[h][a] + al * pv[h][a] + om * sv[h][a]);
                        const cx<T> rn = sv[h][a] - om * tv[h][a];
                        res_st<S>(R, t, c3 + a, rn);
                        res_st<S>(P, t, c3 + a, rn + be * (pv[h][a] - om * vv[h][a]));
                    }
                }
            }
        }
        fence();
    }
    // ---- x64 += |r64| x_l; the states for the outer loop
    if (o.active) {
        const double sc = sqrt(o.r2);
        for (int i = first; i < nit; i += RES_ROUND) {
            const int cb = c0 + i;
            const uint32_t t = res_tile(c0 + i);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const cx<T> x = res_ld<S>(X, t, c3 + a);
                double2 &z = reinterpret_cast<double2 *>(A.x64)[((size_t)cb * 12 + c3 + a) * A.N + rg];
                z = make_double2(z.x + sc * (double)x.re, z.y + sc * (double)x.im);
            }
        }
    }
    if (rank == 0 && tid == 0) A.st[rg] = sh.rhs;
}

}  // namespace dl
