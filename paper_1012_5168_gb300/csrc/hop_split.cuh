// The FP64 Wilson hop with the four direction pairs of an output site on four
// warps, for launches with few sites.
//
// A whole-site thread issues about 870 FP64 instructions, one after the other at
// 17 to 70 cycles each (two FP64 lanes a clock and SM, about 70 cycles latency): a
// launch that leaves an SM with few warps is bound by that chain, not by the
// units.  Here warp q of four takes mu = q, forward and backward, of 32 (site,
// right-hand side) items; the four contributions meet in shared memory, and warp q
// goes on with spin q: 230 instructions a thread, a twentieth more in all.  A block is
// one such group or two (GR; width 64 needs two, for a thread to keep its
// right-hand side).
#pragma once

#include "hop.cuh"

namespace dl {

// Spin MU of mu's contribution in own[], the other spins in part[][lane].
template <int MU>
__device__ __forceinline__ void split_pair_f64(const HopArgs &A, const Site &st, int cb, int r0, cx<double> (&own)[3],
                                               cx<double> (*part)[32], int lane) {
    cx<double> acc[12];
#pragma unroll
    for (int c = 6; c < 12; ++c) acc[c] = zero<double>();
    hop_pair_f64<MU, true>(A, st, cb, r0, acc);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (s == MU) own[a] = acc[3 * s + a];
            else part[(s - (s > MU ? 1 : 0)) * 3 + a][lane] = acc[3 * s + a];
        }
}

// Modes and reductions as hop_kernel<double>.
template <int MODE, int RED, int GR>
__global__ void __launch_bounds__(128 * GR) hop_split_f64_kernel(HopArgs A) {
    constexpr int NV = RedCount<RED>::n > 0 ? RedCount<RED>::n : 1;
    __shared__ cx<double> part[GR][4][9][32];  // [group][mu][other spins][item]
    const int lane = threadIdx.x & 31, grp = (threadIdx.x >> 5) & (GR - 1), q = threadIdx.x / (32 * GR);
    const int lgN = __ffs(A.N) - 1, total = (A.cb_end - A.cb_begin) << lgN;
    const int j = threadIdx.x & (32 * GR - 1) & (A.N - 1);  // items advance by 32 GR, a multiple of N
    const bool on = !A.act || __ldg(A.act + (size_t)j * A.act_stride) != 0;
    const double *yd = reinterpret_cast<const double *>(A.y), *zd = reinterpret_cast<const double *>(A.z);
    const double *rd = reinterpret_cast<const double *>(A.rhat);
    double *od = reinterpret_cast<double *>(A.out);
    cx<double> red[1][NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) red[0][k] = zero<double>();
    for (int base = blockIdx.x * 32 * GR; base < total; base += gridDim.x * 32 * GR) {
        const int i = base + grp * 32 + lane, cb = A.cb_begin + (i >> lgN);
        const bool in = on && i < total;
        cx<double> d[3];
        if (in) {
            const Site st = decode(__ldg(A.coords + (size_t)A.p * A.g.Vh + cb), A.g);
            if (q == 0) split_pair_f64<0>(A, st, cb, j, d, part[grp][0], lane);
            else if (q == 1) split_pair_f64<1>(A, st, cb, j, d, part[grp][1], lane);
            else if (q == 2) split_pair_f64<2>(A, st, cb, j, d, part[grp][2], lane);
            else split_pair_f64<3>(A, st, cb, j, d, part[grp][3], lane);
        }
        __syncthreads();
        if (in) {
#pragma unroll
            for (int m = 1; m < 4; ++m) {
                const int mu = (q + m) & 3, row = (q - (q > mu ? 1 : 0)) * 3;
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] = d[a] + part[grp][mu][row + a][lane];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const size_t off = (((size_t)cb * 12 + 3 * q + a) * A.N + j) * 2;
                cx<double> o = A.c * d[a], y = zero<double>();
                if (MODE != MODE_PLAIN) y = ld_link<double>(yd + off);
                if (MODE == MODE_XPAY) o = y + A.c * d[a];
                if (MODE == MODE_RESID) o = ld_link<double>(zd + off) - y - A.c * d[a];
                *reinterpret_cast<double2 *>(od + off) = make_double2(o.re, o.im);
                if (RED == RED_R0DOT) cjmac(red[0][0], ld_link<double>(rd + off), o);
                if constexpr (RED == RED_BICG) {
                    const cx<double> rh = ld_link<double>(rd + off);
                    cjmac(red[0][0], o, y);
                    norm_mac(red[0][1], o);
                    cjmac(red[0][2], rh, y);
                    cjmac(red[0][3], rh, o);
                    norm_mac(red[0][4], y);
                }
                if (RED == RED_NORM) norm_mac(red[0][0], o);
            }
        }
        __syncthreads();  // part is free again
    }
    if (RED != RED_NONE) block_reduce<1, NV, double>(red, A.N, A.N, A.partials, part);
}

}  // namespace dl
