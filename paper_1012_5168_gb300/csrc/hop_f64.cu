// Wilson-hop instantiations for double storage: FP64 arithmetic, and float-float
// arithmetic (hop_ff.cuh) for the defect-correction steps of mixed-precision solves.
#include "hop_ff.cuh"
#include "hop_split.cuh"
#include "launch.h"

namespace dl {

template <int R, int MODE, int RED>
static cudaError_t go(const HopArgs &a, Launch &l) {
    if (a.clovinv) {  // clover: A^-1 of the output site in the epilogue
        clamp_grid(l, resident_blocks(hop_kernel_clov<double, MODE, RED>, l.block, l.smem));
        hop_kernel_clov<double, MODE, RED><<<l.grid, l.block, l.smem, l.stream>>>(a);
        return cudaGetLastError();
    }
    // Where every SM gets at most one block of 64 (site, right-hand side) items, four warps
    // share 32 of them (hop_split.cuh), one group a block while that fills no more than the
    // SMs: plain hops of 12.4 us (up to 32 items an SM) and 20.5 us (64) against 33 us for
    // any number of sites up to 100 an SM; at 108 items an SM both take 35 us.
    const long items = (long)(a.cb_end - a.cb_begin) * a.N;
    if (l.num_sms > 0 && items <= 64L * l.num_sms) {
        const int groups = a.N <= 32 && items <= 32L * l.num_sms ? 1 : 2;
        auto kernel = groups == 1 ? hop_split_f64_kernel<MODE, RED, 1> : hop_split_f64_kernel<MODE, RED, 2>;
        l.block = 128 * groups;
        l.smem = 0;
        l.grid = (int)((items + 32 * groups - 1) / (32 * groups));
        kernel<<<l.grid, l.block, 0, l.stream>>>(a);
        return cudaGetLastError();
    }
    // 168 registers let six blocks of 64 threads share an SM (about 180: five).  One right-hand
    // side on 16^3 x 32: 115 / 121 / 141 us (plain, <rhat, v>, five sums) against 124 / 131 / 152.
    // Beyond one round the blocks with a second item lie on some SMs and not on others.  With 7.5 to
    // 10.5 blocks an SM (of any residency) that leaves six at once behind five: 8.0 blocks, plain hop, 145
    // against 125 us, 9.5 blocks 181 / 156, at 7.2 and 10.5 both alike; from two rounds on six are ahead
    // by 4% (14.2 blocks) or behind by 5% (16.4) and mostly alike.
    const bool five = l.block == 64 && 2L * l.grid > 15L * l.num_sms && 2L * l.grid <= 21L * l.num_sms;
    auto kernel = five ? hop_kernel<double, R, MODE, RED> : hop_kernel_cap<double, R, MODE, RED, 168>;
    clamp_grid(l, resident_blocks(kernel, l.block, l.smem));
    kernel<<<l.grid, l.block, l.smem, l.stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_hop_f64(int R, int mode, int red, const HopArgs &a, Launch &l) {
#define DL_CASE(r, m, rd) \
    if (R == r && mode == m && red == rd) return go<r, m, rd>(a, l);
    DL_CASE(1, MODE_PLAIN, RED_NONE)
    DL_CASE(1, MODE_XPAY, RED_NONE)
    DL_CASE(1, MODE_XPAY, RED_R0DOT)
    DL_CASE(1, MODE_XPAY, RED_BICG)
    DL_CASE(1, MODE_XPAY, RED_NORM)
    DL_CASE(1, MODE_RESID, RED_NORM)
#undef DL_CASE
    return cudaErrorInvalidValue;
}

template <int MODE, int RED, bool YFF, bool OFF>
static cudaError_t go_ff(const HopArgs &a, Launch &l) {
    clamp_grid(l, resident_blocks(hop_ff_rows_kernel<MODE, RED, YFF, OFF>, l.block, l.smem));
    hop_ff_rows_kernel<MODE, RED, YFF, OFF><<<l.grid, l.block, l.smem, l.stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_hop_ff(int mode, int red, int fmt, const HopArgs &a, Launch &l) {
    const bool yff = fmt & FF_Y, off = fmt & FF_OUT;
#define DL_CASE(m, rd, y, o) \
    if (mode == m && red == rd && yff == y && off == o) return go_ff<m, rd, y, o>(a, l);
    DL_CASE(MODE_PLAIN, RED_NONE, false, false)
    DL_CASE(MODE_XPAY, RED_NONE, false, false)
    DL_CASE(MODE_XPAY, RED_NONE, true, false)
    DL_CASE(MODE_XPAY, RED_NONE, true, true)
    DL_CASE(MODE_XPAY, RED_NORM, false, false)
    DL_CASE(MODE_RESID, RED_NORM, true, false)
#undef DL_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_ff_cast(const double *src, double *dst, size_t n_complex, int to_ff, int grid, cudaStream_t s) {
    ff_cast_kernel<<<grid, 256, 0, s>>>(src, dst, (long)n_complex, to_ff);
    return cudaGetLastError();
}

}  // namespace dl
