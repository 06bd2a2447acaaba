// Momentum projection and two-point functions (Sec. 3, Eqs. 1 and 3).
//
// Loops at spatial momentum p = 2 pi n / L (n integer):
//     L_Gamma(p, t) = sum_{x in t} exp(-i p.(x - o)) eta(x)^dag Gamma phi(x),
// and the connected meson function of a point source at y (o = y):
//     C^{BA}(p, t) = - sum_x exp(-i p.(x - y)) Tr[g5 S(x)^dag g5 Gamma_B S(x) Gamma_A].
// Both run in three steps: a per-site matrix (the 4x4 spin matrix
// phi eta^dag summed over a group of pairs, or the hermitian 16x16 colour-summed
// product of the propagator with its conjugate), its Fourier sums over each
// timeslice against a phase table, and the Gamma traces.  All sums are FP64 in a fixed order.  The disconnected
// function combines per-noise loops at p and -p over pairs of distinct noise
// vectors, so no noise vector is multiplied with itself.
#pragma once

#include "common.cuh"

namespace dl {

// ph[q][s] = exp(-i 2 pi sum_i n_i (x_i - o_i) / L_i), s = x + Lx (y + Ly z).
static __global__ void phase_table_kernel(double2 *ph, const int *mom, int n_mom, Geom g, int ox, int oy, int oz) {
    const int V3 = g.L[0] * g.L[1] * g.L[2];
    const int total = n_mom * V3;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int q = idx / V3, s = idx % V3;
        const int x = s % g.L[0], y = (s / g.L[0]) % g.L[1], z = s / (g.L[0] * g.L[1]);
        const int kx = ((mom[3 * q] * (x - ox)) % g.L[0] + g.L[0]) % g.L[0];
        const int ky = ((mom[3 * q + 1] * (y - oy)) % g.L[1] + g.L[1]) % g.L[1];
        const int kz = ((mom[3 * q + 2] * (z - oz)) % g.L[2] + g.L[2]) % g.L[2];
        const double frac = (double)kx / g.L[0] + (double)ky / g.L[1] + (double)kz / g.L[2];
        double sn, cs;
        sincospi(-2.0 * frac, &sn, &cs);
        ph[idx] = make_double2(cs, sn);
    }
}

struct SiteSpinArgs {
    const double *eta;  // EO tile [2][Vh][12][N]
    const double *phi;
    const uint32_t *coords;
    Geom g;
    int N, n;           // layout width, right-hand sides in use
    int t_lo, nt;       // timeslices t_lo .. t_lo + nt - 1 (nt = 1 with tcol)
    const int *tcol;    // if set: right-hand side j lives on timeslice tcol[j]
    double2 *out;       // [n][nt][16][V3]: S_{beta alpha}(x) = sum_a phi_{beta a}(x) conj(eta_{alpha a}(x))
};

// One thread per (site of the timeslice, right-hand side); j is the fastest
// index so that a warp reads contiguous right-hand sides of the EO tile.
static __global__ void site_spin_kernel(SiteSpinArgs A) {
    const int V3 = A.g.L[0] * A.g.L[1] * A.g.L[2];
    const long total = (long)A.nt * 2 * A.g.V3h * A.n;
    const size_t half = (size_t)A.g.Vh * 12 * A.N * 2;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int j = (int)(idx % A.n);
        const long sp = idx / A.n;
        const int cbl = (int)(sp % A.g.V3h);
        const int p = (int)((sp / A.g.V3h) % 2);
        const int tt = (int)(sp / (2L * A.g.V3h));
        const int t = A.tcol ? A.tcol[j] : A.t_lo + tt;
        const int cb = t * A.g.V3h + cbl;
        const Site st = decode(__ldg(A.coords + (size_t)p * A.g.Vh + cb), A.g);
        const int s = st.c[0] + A.g.L[0] * (st.c[1] + A.g.L[1] * st.c[2]);
        const size_t base = (size_t)p * half + (size_t)cb * 12 * A.N * 2 + (size_t)j * 2;
        cx<double> e[12], f[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            cx<double> v[1];
            ld_pack<double, 1, true>(A.eta + base + (size_t)c * A.N * 2, v);
            e[c] = v[0];
            ld_pack<double, 1, true>(A.phi + base + (size_t)c * A.N * 2, v);
            f[c] = v[0];
        }
        double2 *o = A.out + ((size_t)j * A.nt + tt) * 16 * V3 + s;
#pragma unroll
        for (int be = 0; be < 4; ++be)
#pragma unroll
            for (int al = 0; al < 4; ++al) {
                cx<double> acc = zero<double>();
#pragma unroll
                for (int a = 0; a < 3; ++a) cjmac(acc, e[3 * al + a], f[3 * be + a]);
                o[(size_t)(be * 4 + al) * V3] = make_double2(acc.re, acc.im);
            }
    }
}

// site[g] = sum of the site matrices of each run of `group` right-hand sides (fixed order,
// in place: slot g lies in a group that is summed no later than g).
static __global__ void group_site_kernel(double2 *site, long per, int ng, int group) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < per; i += (long)gridDim.x * blockDim.x)
        for (int g = 0; g < ng; ++g) {
            double re = 0.0, im = 0.0;
            for (int k = 0; k < group; ++k) {
                const double2 v = site[(size_t)(g * group + k) * per + i];
                re += v.x;
                im += v.y;
            }
            site[(size_t)g * per + i] = make_double2(re, im);
        }
}

// Site matrices of a whole group of pairs straight from canonical fields:
//   out[g][tt][16][V3] = sum_{j in group g} sum_a phi_{beta a}(x) conj(eta_{alpha a}(x)).
// Everything after it is linear, so summing the group's pairs here divides the
// Fourier sums and their input by the group size, and no field is converted.
//
// A block of eight warps takes 32 sites and walks the group's pairs: both fields'
// tiles ([32][12] complex, one contiguous run each) go through shared memory, the
// next pair's loads in flight while the current one is multiplied.  Warp w works
// for source spin w & 3 and, of every pair of neighbouring sites, the one of parity
// w >> 2; a lane for (site, beta), so the three products of a colour are one
// warp-wide decision: where a diluted eta vanishes for the whole warp the FP64
// work is left out (dense fields are bound by FP64: 192 FMA a site and pair, 1.2 ms
// for 48 pairs on 16^3 x 32; diluted ones by shared memory, 0.65 ms, where reading the
// fields takes 0.36: all warps read f for every colour, and sites lie 384 bytes apart), except
// that a non-finite phi still makes the sum NaN, as 0 times it would.
struct CanonSpinArgs {
    const double2 *eta, *phi;  // canonical [n][V][12]
    Geom g;
    int V3, group, nt;         // pairs per block; nt timeslices from 0, or (tgrp) one timeslice per group
    int parts;                 // blocks that share a group's pairs: gridDim.z = groups x parts = slots of out
    const int *tgrp;
    double2 *out;
};
__device__ __forceinline__ bool cx_nonzero(double2 z) {
    return (((unsigned)__double2hiint(z.x) | (unsigned)__double2hiint(z.y)) << 1 | (unsigned)__double2loint(z.x) |
            (unsigned)__double2loint(z.y)) != 0u;
}
__device__ __forceinline__ bool cx_bad(double2 z) {  // infinite or NaN, without FP64 instructions
    return (__double2hiint(z.x) & 0x7ff00000) == 0x7ff00000 || (__double2hiint(z.y) & 0x7ff00000) == 0x7ff00000;
}
static __global__ void __launch_bounds__(256) canon_spin_kernel(CanonSpinArgs A) {
    __shared__ double2 se[2][384], sf[2][384];
    const int tile = blockIdx.x, tt = blockIdx.y, gi = blockIdx.z;
    const int t = A.tgrp ? A.tgrp[gi / A.parts] : tt;
    const int s0 = tile * 32, ns = min(32, A.V3 - s0);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, al = w & 3, par = w >> 2, be = lane & 3;
    const long V = (long)A.V3 * A.g.L[3];
    const size_t first = ((size_t)gi * A.group * V + (size_t)t * A.V3 + s0) * 12;
    // the two sites of this lane: of the pairs lane / 4 and lane / 4 + 8, the one of parity par
    int site[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int m = (lane >> 2) + 8 * h, i0 = t * A.V3 + s0 + 2 * m;
        const int y = i0 / A.g.L[0], z = y / A.g.L[1], u = z / A.g.L[2];  // (x of an even site is even)
        site[h] = 2 * m + ((par + y + z + u) & 1);
    }
    cx<double> acc[2] = {zero<double>(), zero<double>()};
    bool bad = false;
    const int ne = ns * 12;  // 384 elements a tile: thread k loads elements k and k + 256 of both fields
    double2 r[4];
    auto load = [&](int j) {
        const size_t o = first + (size_t)j * V * 12;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = threadIdx.x + 256 * h;
            if (k < ne) {
                r[2 * h] = __ldg(A.eta + o + k);
                r[2 * h + 1] = __ldg(A.phi + o + k);
            }
        }
    };
    load(0);
    for (int j = 0; j < A.group; ++j) {
        const int b = j & 1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = threadIdx.x + 256 * h;
            if (k < ne) {
                se[b][k] = r[2 * h];
                sf[b][k] = r[2 * h + 1];
            }
        }
        __syncthreads();  // (buffer b was last read two steps ago, before the previous barrier)
        if (j + 1 < A.group) load(j + 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool in = site[h] < ns;
            const int o = (in ? site[h] : 0) * 12;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double2 e = se[b][o + 3 * al + a], f = sf[b][o + 3 * be + a];
                if (__any_sync(0xffffffffu, in && cx_nonzero(e)))
                    cjmac(acc[h], mk(e.x, e.y), mk(f.x, f.y));
                else
                    bad |= in && cx_bad(f);
            }
        }
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    double2 *o = A.out + (((size_t)gi * A.nt + tt) * 16 + be * 4 + al) * A.V3 + s0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (site[h] < ns) o[site[h]] = bad ? make_double2(nan, nan) : make_double2(acc[h].re, acc[h].im);
}

struct __align__(16) FourierSum {
    double x, y, z, w;  // sums of c x, s y, c y, s x
};

// Fourier sums over a timeslice.  Momenta come as representatives r with
// phases e^{-i p.x} = c + i s; p and -p share one (conjugate phases), and the four
// real sums
//   out[row][r] = (sum c x, sum s y, sum c y, sum s x)   of  z = x + i y = in[row][site]
// give the sums of z and of conj(z) at p and at -p.  in: [rows][V3] (a row is one
// matrix entry on one timeslice).  A warp takes a row and up to four representatives
// (blockIdx.y picks which): its lanes walk the sites (coalesced).  At the end the lanes
// exchange halves of their 16 sums instead of each adding all of them, 16 FP64
// additions a warp instead of 80.  Bound by FP64: 3072 rows and 172 representatives of 4096 sites
// are 13.9 ms of FMA, and the loops of 24 pairs that ask for them take 15.1 ms.  (Two rows a
// warp, each phase loaded once for both: slower.)  A lone representative of zero momentum (zero[r0])
// needs sums of x and y only; among others its phases are ones and zeros like any: told apart in
// the loop, the compiler issued both kinds of sums, half as many FP64 instructions again (23.9 ms).
static __global__ void __launch_bounds__(128) fourier_kernel(const double2 *in, const double2 *ph, const int *zero,
                                                             int V3, long rows, int n_rep, FourierSum *out) {
    const int lane = threadIdx.x & 31;
    const long row = (long)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int r0 = blockIdx.y * 4;
    if (row >= rows) return;
    double acc[16];  // [4 representative + sum]
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.0;
    const double2 *src = in + (size_t)row * V3;
    if (n_rep - r0 == 1 && zero[r0]) {
        for (int s = lane; s < V3; s += 32) {
            const double2 v = __ldg(src + s);
            acc[0] += v.x;
            acc[2] += v.y;
        }
    } else {
        const double2 *w_[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w_[r] = ph + (size_t)min(r0 + r, n_rep - 1) * V3;
        for (int s = lane; s < V3; s += 32) {
            const double2 v = __ldg(src + s);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (r0 + r >= n_rep) break;
                const double2 w = __ldg(w_[r] + s);
                acc[4 * r] = ::fma(w.x, v.x, acc[4 * r]);
                acc[4 * r + 1] = ::fma(w.y, v.y, acc[4 * r + 1]);
                acc[4 * r + 2] = ::fma(w.x, v.y, acc[4 * r + 2]);
                acc[4 * r + 3] = ::fma(w.y, v.x, acc[4 * r + 3]);
            }
        }
    }
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {  // the lanes with bit 2 h set keep the upper h sums
        const bool up = (lane & (2 * h)) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k)
            acc[k] = (up ? acc[h + k] : acc[k]) + __shfl_xor_sync(0xffffffffu, up ? acc[k] : acc[h + k], 2 * h);
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    const int k = lane >> 1;  // the sum that this lane holds
    if ((lane & 1) == 0 && r0 + (k >> 2) < n_rep) reinterpret_cast<double *>(out + (size_t)row * n_rep + r0)[k] = acc[0];
}
// sum of e^{-i p.x} z (CONJ: of e^{-i p.x} conj(z)) from the four sums; sg = -1: at -p.
template <bool CONJ> __device__ __forceinline__ double2 fourier_value(FourierSum f, int sg) {
    const double s = sg < 0 ? -1.0 : 1.0;
    return CONJ ? make_double2(f.x + s * f.y, s * f.w - f.z) : make_double2(f.x - s * f.y, f.z + s * f.w);
}

// L_Gamma(p, t) = sum_{alpha beta} Gamma_{alpha beta} S_{beta alpha}(p, t):
// F [n][nt][16][n_rep] -> out[j][q][G][T] at t = tcol[j] or t_lo + tt; momentum q is
// representative rep[q] >> 1, negated if rep[q] & 1.
static __global__ void mom_gamma_kernel(const FourierSum *F, const double2 *gammas, const int *rep, int n_rep, int n,
                                        int nt, int Q, int T, int t_lo, const int *tcol, double2 *out) {
    const int total = n * nt * Q * 16;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int G = idx % 16;
        const int q = (idx / 16) % Q;
        const int tt = (idx / (16 * Q)) % nt;
        const int j = idx / (16 * Q * nt);
        const FourierSum *f = F + ((size_t)j * nt + tt) * 16 * n_rep + (rep[q] >> 1);
        const int sg = (rep[q] & 1) ? -1 : 1;
        double re = 0.0, im = 0.0;
        for (int al = 0; al < 4; ++al)
            for (int be = 0; be < 4; ++be) {
                const double2 gm = gammas[(G * 4 + al) * 4 + be];
                if (gm.x == 0.0 && gm.y == 0.0) continue;
                const double2 v = fourier_value<false>(f[(size_t)(be * 4 + al) * n_rep], sg);
                re += gm.x * v.x - gm.y * v.y;
                im += gm.x * v.y + gm.y * v.x;
            }
        const int t = tcol ? tcol[j] : t_lo + tt;
        out[(((size_t)j * Q + q) * 16 + G) * T + t] = make_double2(re, im);
    }
}

// The point-source propagator's products P_{(beta alpha),(beta' alpha')}(x) =
// sum_{a,b} conj(S_{beta b, alpha a}) S_{beta' b, alpha' a} form a hermitian 16 x 16
// matrix: 136 entries (beta, alpha) <= (beta', alpha').  Entry number: 40 of the
// diagonal blocks beta = beta' (10 each), then 6 blocks beta < beta' of 16.
constexpr int MESON_E = 136;
__host__ __device__ __forceinline__ int meson_entry(int be, int al, int be2, int al2) {  // (be, al) <= (be2, al2)
    if (be == be2) return be * 10 + al * 4 - al * (al - 1) / 2 + (al2 - al);
    return 40 + (be * (7 - be) / 2 + (be2 - be - 1)) * 16 + al * 4 + al2;
}

// prop: canonical [12][V][4][3], column j = 3 alpha + a; out [t][136][V3].  A block
// stages the 144 components of 32 sites in shared memory (one contiguous run a
// column) and gives each of its ten warps one block (beta, beta') of the matrix, a
// lane per site.  Bound by FP64 (4896 FMA a site, 1.0 ms on 16^3 x 32; all 256
// entries took 1.95 ms): the hermitian half is all that is formed, and stored
// entry-major so that lanes write, and the Fourier sums read, contiguous sites.
// prop may lie on any 8-byte boundary: one that is not a 16-byte boundary (AL16 false) is
// read a double at a time.
template <bool AL16>
static __global__ void __launch_bounds__(320) meson_site_kernel(const double *prop, int V, int V3, double2 *out) {
    extern __shared__ double2 msm[];  // [144][33]
    const int s0 = blockIdx.x * 32, ns = min(32, V - s0);
    for (int k = threadIdx.x; k < 12 * 384; k += 320) {
        const int col = k / 384, e = k - col * 384, site = e / 12, c = e - site * 12;
        const double *v = prop + (((size_t)col * V + s0) * 12 + e) * 2;
        if (site < ns)
            msm[(col * 12 + c) * 33 + site] =
                AL16 ? __ldg(reinterpret_cast<const double2 *>(v)) : make_double2(__ldg(v), __ldg(v + 1));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane >= ns) return;
    const int i = s0 + lane;
    double2 *o = out + (size_t)(i / V3) * MESON_E * V3 + i % V3;
    auto S = [&](int be, int b, int al, int a) {
        const double2 v = msm[((3 * al + a) * 12 + 3 * be + b) * 33 + lane];
        return mk(v.x, v.y);
    };
    cx<double> acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = zero<double>();
    if (w < 4) {
        for (int ab = 0; ab < 9; ++ab) {
            const int a = ab / 3, b = ab % 3;
            cx<double> u[4];
#pragma unroll
            for (int al = 0; al < 4; ++al) u[al] = S(w, b, al, a);
#pragma unroll
            for (int al = 0; al < 4; ++al)
#pragma unroll
                for (int al2 = al; al2 < 4; ++al2) cjmac(acc[al * 4 + al2], u[al], u[al2]);
        }
#pragma unroll
        for (int al = 0; al < 4; ++al)
#pragma unroll
            for (int al2 = al; al2 < 4; ++al2)
                o[(size_t)meson_entry(w, al, w, al2) * V3] = make_double2(acc[al * 4 + al2].re, acc[al * 4 + al2].im);
    } else {
        const int p = w - 4, be = p < 3 ? 0 : (p < 5 ? 1 : 2), be2 = p < 3 ? p + 1 : (p < 5 ? p - 1 : 3);
        for (int ab = 0; ab < 9; ++ab) {
            const int a = ab / 3, b = ab % 3;
            cx<double> u[4], v[4];
#pragma unroll
            for (int al = 0; al < 4; ++al) {
                u[al] = S(be, b, al, a);
                v[al] = S(be2, b, al, a);
            }
#pragma unroll
            for (int al = 0; al < 4; ++al)
#pragma unroll
                for (int al2 = 0; al2 < 4; ++al2) cjmac(acc[al * 4 + al2], u[al], v[al2]);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k)
            o[(size_t)meson_entry(be, k / 4, be2, k % 4) * V3] = make_double2(acc[k].re, acc[k].im);
    }
}

// C^{BA}(q, t - t_src) = - sum g5_alpha g5_beta (Gamma_B)_{beta beta'} (Gamma_A)_{alpha' alpha}
//                          F_t[q][(beta alpha),(beta' alpha')];  F [T][136][n_rep], out [Q][16 A][16 B][T].
// Every Gamma of the basis has one non-zero entry per row (its column and value
// are looked up once per block), so an output is a sum of 16 terms.
static __global__ void __launch_bounds__(256) meson_gamma_kernel(const FourierSum *F, const double2 *gammas, const int *rep,
                                                                 int n_rep, int T, int Q, int t_src, double2 *out) {
    __shared__ double2 val[16][4];
    __shared__ int col[16][4];
    for (int k = threadIdx.x; k < 64; k += blockDim.x) {
        int c = 0;
        for (int m = 1; m < 4; ++m)
            if (gammas[k * 4 + m].x != 0.0 || gammas[k * 4 + m].y != 0.0) c = m;
        col[k / 4][k % 4] = c;
        val[k / 4][k % 4] = gammas[k * 4 + c];
    }
    __syncthreads();
    const int total = Q * 256 * T;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int t = idx % T;
        const int B = (idx / T) % 16;
        const int A = (idx / (16 * T)) % 16;
        const int q = idx / (256 * T);
        const FourierSum *f = F + (size_t)t * MESON_E * n_rep + (rep[q] >> 1);
        const int sg = (rep[q] & 1) ? -1 : 1;
        double re = 0.0, im = 0.0;
        for (int be = 0; be < 4; ++be)
            for (int al2 = 0; al2 < 4; ++al2) {
                const int be2 = col[B][be], al = col[A][al2];
                const double2 gb = val[B][be], ga = val[A][al2];
                const double sn = ((al < 2) == (be < 2)) ? 1.0 : -1.0;  // g5_alpha g5_beta
                const double2 g = make_double2(sn * (gb.x * ga.x - gb.y * ga.y), sn * (gb.x * ga.y + gb.y * ga.x));
                const bool lower = be * 4 + al > be2 * 4 + al2;
                const double2 v = lower ? fourier_value<true>(f[(size_t)meson_entry(be2, al2, be, al) * n_rep], sg)
                                        : fourier_value<false>(f[(size_t)meson_entry(be, al, be2, al2) * n_rep], sg);
                re += g.x * v.x - g.y * v.y;
                im += g.x * v.y + g.y * v.x;
            }
        out[(((size_t)q * 16 + A) * 16 + B) * T + (t - t_src + T) % T] = make_double2(-re, -im);
    }
}

// D^{BA}(q, dt) = -(1/(V3 T)) sum_t E[L_B(q, t + dt) L_A(-q, t)], the expectation over
// pairs of distinct noise vectors n != m that cover t + dt and t respectively:
//   E = [(sum_{n in C(t+dt)} L_B^n)(sum_{m in C(t)} L_A^m) - sum_{n in both} L_B^n L_A^n]
//       / (|C(t+dt)| |C(t)| - |C(t+dt) and C(t)|).
// L [n][Q][16][T], cover [n][T] (1: the noise vector's loop covers t), minus [Q].
static __global__ void disconnected_kernel(const double2 *L, const unsigned char *cover, const int *minus, int n, int Q,
                                           int T, double norm, double2 *out) {
    const int total = Q * 256 * T;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int dt = idx % T;
        const int B = (idx / T) % 16;
        const int A = (idx / (16 * T)) % 16;
        const int q = idx / (256 * T);
        const int qm = minus[q];
        double re = 0.0, im = 0.0;
        for (int t = 0; t < T; ++t) {
            const int t2 = (t + dt) % T;
            double xr = 0, xi = 0, yr = 0, yi = 0, zr = 0, zi = 0;
            long c1 = 0, c2 = 0, c12 = 0;
            for (int k = 0; k < n; ++k) {
                const bool in1 = cover[(size_t)k * T + t2] != 0, in2 = cover[(size_t)k * T + t] != 0;
                if (!in1 && !in2) continue;
                const double2 lb = L[(((size_t)k * Q + q) * 16 + B) * T + t2];
                const double2 la = L[(((size_t)k * Q + qm) * 16 + A) * T + t];
                if (in1) { xr += lb.x; xi += lb.y; ++c1; }
                if (in2) { yr += la.x; yi += la.y; ++c2; }
                if (in1 && in2) {
                    zr += lb.x * la.x - lb.y * la.y;
                    zi += lb.x * la.y + lb.y * la.x;
                    ++c12;
                }
            }
            const long pairs = c1 * c2 - c12;
            if (pairs <= 0) continue;
            re += ((xr * yr - xi * yi) - zr) / (double)pairs;
            im += ((xr * yi + xi * yr) - zi) / (double)pairs;
        }
        out[idx] = make_double2(-norm * re, -norm * im);
    }
}

}  // namespace dl
