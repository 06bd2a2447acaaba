// Launch of one Wilson-hop instantiation for a low-precision storage type S
// (float or bf16): the kernel kind picks the direct, prefetching, staged or
// blocked-mapping, warp-staged or (BF16 only) tensor-core kernel.  hop_f32*.cu
// and hop_bf16*.cu instantiate it.  The
// one-time settings (shared-memory opt-ins, the blocked kernel's block shape)
// are guarded so that contexts used from several host threads can launch
// concurrently.
#pragma once

#include <algorithm>
#include <mutex>

#include <type_traits>

#include "hop_mma.cuh"
#include "launch.h"

namespace dl {

// Raise a kernel's dynamic shared-memory limit to at least `smem` (beyond the
// default 48 KiB), once per larger request.
template <typename K>
inline cudaError_t opt_in_smem(K kernel, size_t smem, size_t &opted, std::mutex &m) {
    if (smem <= 48 * 1024) return cudaSuccess;
    std::lock_guard<std::mutex> g(m);
    if (smem <= opted) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) opted = smem;
    return e;
}

// Blocks per SM of a warp-staged kernel.  Its sites are dealt out to the warps of the whole
// grid, so every block has to be resident.  The occupancy query counts all 228 kB of shared
// memory, but the launch may be given the next smaller split with L1, 196 kB.  Which one
// follows from how much of the larger split's blocks the smaller one holds: with 6 of 7
// (plain hop, FP32, kind 11, width 32: seven blocks of 30,464 bytes, 1 kB of it the system's) six ran together,
// the seventh after them (0.248 ms on 16^3 x 32 against 0.121 with six); with 5 of 6 (kind
// 12) and 3 of 4 (kind 4 at width 32, kind 11 at width 64: 94 us against 100 with three
// on 16 x 20 x 8 x 22) the larger one.  Hence the line at 0.85.
template <typename K> int ws_blocks(K kern, int block, size_t smem) {
    const int small = (int)(196 * 1024 / (smem + 1024)), large = (int)(228 * 1024 / (smem + 1024));
    const int fit = 20 * small >= 17 * large ? small : large;
    return std::min(std::min(resident_blocks(kern, block, smem), std::max(fit, 1)), 16);
}

// Warp-staged hop (hop_ws.cuh): NSTO stages (0: as many as suit the width), SPW sites of 32 R / SPW
// right-hand sides per warp.  Evict-first streams (a.stream) in FP32 where they gain: 24^3 x 48,
// width 32, fused hops of kinds 4 and 11 907 -> 842 and 907 -> 777 us, plain hop of kind 11
// 581 -> 570; width 16 (kind 12) fused 420 -> 406, plain 303 -> 305; 24 x 16 x 8 x 40, width 64,
// fused 282 -> 275, plain 194 both.  BF16: 843 -> 847 and 920 -> 938 fused.
template <typename S, int R, int MODE, int RED, int NSTO, int SPW, bool CLOV, bool EF>
cudaError_t go_ws_ef(const HopArgs &a, Launch &l) {
    static size_t opted = 0;
    static std::mutex m;
    auto kern = hop_kernel_ws<S, R, MODE, RED, NSTO, SPW, CLOV, EF>;
    l.block = WS_WARPS * 32;
    l.smem = WsShape<S, R, NSTO, SPW, CLOV>::WB * WS_WARPS;
    const cudaError_t e = opt_in_smem(kern, l.smem, opted, m);
    if (e != cudaSuccess) return e;
    l.grid = (l.num_sms > 0 ? l.num_sms : 1) * ws_blocks(kern, l.block, l.smem);
    kern<<<l.grid, l.block, l.smem, l.stream>>>(a);
    return cudaGetLastError();
}
template <typename S, int R, int MODE, int RED, int NSTO, int SPW = 1, bool CLOV = false>
cudaError_t go_ws(const HopArgs &a, Launch &l) {
    if (a.N != 32 * R / SPW) return cudaErrorInvalidValue;
    if constexpr (std::is_same<S, float>::value && (RED != RED_NONE || (R == 1 && SPW == 1 && NSTO == 2)))
        if (a.stream) return go_ws_ef<S, R, MODE, RED, NSTO, SPW, CLOV, true>(a, l);
    return go_ws_ef<S, R, MODE, RED, NSTO, SPW, CLOV, false>(a, l);
}

template <typename S, int R, int MODE, int RED>
cudaError_t go_hop(const HopArgs &a, Launch &l, int kind) {
    if (a.clovinv) {  // clover: A^-1 in the epilogue, one right-hand side per thread
        if constexpr (R == 1) {
            // FP32, widths 32 and 16: warp-staged, A^-1 copied in with the links.  16^3 x 32,
            // width 32: 136 us plain, 158 and 173 fused, where the direct kernel with its
            // 1152 bytes of links and A^-1 per thread took 147, 203 and 216.
            if constexpr (std::is_same<S, float>::value) {
                if (a.N == 32) return go_ws<S, 1, MODE, RED, 2, 1, true>(a, l);
                if (a.N == 16) return go_ws<S, 1, MODE, RED, 2, 2, true>(a, l);
            }
            clamp_grid(l, resident_blocks(hop_kernel_clov<S, MODE, RED>, l.block, l.smem));
            hop_kernel_clov<S, MODE, RED><<<l.grid, l.block, l.smem, l.stream>>>(a);
            return cudaGetLastError();
        }
        return cudaErrorInvalidValue;
    }
    constexpr int cap = HopRegCap<S, R, MODE, RED>::n;
    auto direct = [] {
        if constexpr (cap > 0) return hop_kernel_cap<S, R, MODE, RED, cap>;
        else return hop_kernel<S, R, MODE, RED>;
    }();
    if (kind == 0) {
        if constexpr (cap > 0) {
            if (a.N == 32 || a.N == 16) {  // the usual widths: offsets as compile-time constants
                auto k = a.N == 32 ? hop_kernel_cap<S, R, MODE, RED, cap, 32> : hop_kernel_cap<S, R, MODE, RED, cap, 16>;
                clamp_grid(l, resident_blocks(k, l.block, l.smem));
                k<<<l.grid, l.block, l.smem, l.stream>>>(a);
                return cudaGetLastError();
            }
        }
        clamp_grid(l, resident_blocks(direct, l.block, l.smem));
        direct<<<l.grid, l.block, l.smem, l.stream>>>(a);
        return cudaGetLastError();
    }
    if (kind == 10) {  // the direct FP32 kernel under a wider register cap (80 plain, 96 fused)
        if constexpr (std::is_same<S, float>::value && R == 1) {
            constexpr int wcap = MODE == MODE_PLAIN ? 80 : 96;
            auto k = a.N == 32   ? hop_kernel_cap<S, 1, MODE, RED, wcap, 32>
                     : a.N == 16 ? hop_kernel_cap<S, 1, MODE, RED, wcap, 16>
                                 : hop_kernel_cap<S, 1, MODE, RED, wcap>;
            clamp_grid(l, resident_blocks(k, l.block, l.smem));
            k<<<l.grid, l.block, l.smem, l.stream>>>(a);
            return cudaGetLastError();
        }
        return cudaErrorInvalidValue;
    }
    if (kind == 1) {
        static size_t opted = 0;
        static std::mutex m;
        const cudaError_t e = opt_in_smem(hop_kernel_pf<S, R, MODE, RED>, l.smem, opted, m);
        if (e != cudaSuccess) return e;
        hop_kernel_pf<S, R, MODE, RED><<<l.grid, l.block, l.smem, l.stream>>>(a);
        return cudaGetLastError();
    }
    if (kind == 2) {
        static size_t opted = 0;
        static std::mutex m;
        const cudaError_t e = opt_in_smem(hop_kernel_tma<S, R, MODE, RED, TMA_STAGES>, l.smem, opted, m);
        if (e != cudaSuccess) return e;
        hop_kernel_tma<S, R, MODE, RED, TMA_STAGES><<<l.grid, l.block, l.smem, l.stream>>>(a);
        return cudaGetLastError();
    }
    if (kind == 3) {
        constexpr int NV = RedCount<RED>::n;
        const int G = a.N / R;
        const size_t per_warp = NV ? (size_t)(G < 32 ? G : 32) * R * NV * sizeof(cx<float>) : 0;
        // block shape for the G last seen: block | resident << 16 | G << 24
        static std::atomic<uint32_t> shape{0};
        uint32_t sh = shape.load(std::memory_order_relaxed);
        if (sh == 0 || (int)(sh >> 24) != G) {
            int res = 1;
            const int blk = widest_block(direct, G > 32 ? G : 32, per_warp, &res);
            sh = (uint32_t)blk | ((uint32_t)(res < 16 ? res : 16) << 16) | ((uint32_t)G << 24);
            shape.store(sh, std::memory_order_relaxed);
        }
        HopArgs b = a;
        b.blocked = 1;
        l.block = (int)(sh & 0xffff);
        l.smem = per_warp * (l.block / 32);
        l.grid = (l.num_sms > 0 ? l.num_sms : 1) * (int)((sh >> 16) & 0xff);
        direct<<<l.grid, l.block, l.smem, l.stream>>>(b);
        return cudaGetLastError();
    }
    if (kind == 4) return go_ws<S, R, MODE, RED, 0>(a, l);  // warp-staged: one site per warp, so N = 32 R
    if (kind == 11) return go_ws<S, R, MODE, RED, 2>(a, l);  // the same with two stages
    if (kind == 12) {  // at width 16, two sites per warp (FP32), two stages
        if constexpr (std::is_same<S, float>::value && R == 1) return go_ws<S, 1, MODE, RED, 2, 2>(a, l);
        return cudaErrorInvalidValue;
    }
    if (kind == 6) {  // direct loads, packed FP32 arithmetic (FP32 storage, R = 1)
        if constexpr (std::is_same<S, float>::value && R == 1) {
            constexpr int xcap = MODE == MODE_PLAIN ? 64 : 72;
            if (a.N == 32) {
                clamp_grid(l, resident_blocks(hop_kernel_x2<MODE, RED, xcap, 32>, l.block, l.smem));
                hop_kernel_x2<MODE, RED, xcap, 32><<<l.grid, l.block, l.smem, l.stream>>>(a);
            } else {
                clamp_grid(l, resident_blocks(hop_kernel_x2<MODE, RED, xcap>, l.block, l.smem));
                hop_kernel_x2<MODE, RED, xcap><<<l.grid, l.block, l.smem, l.stream>>>(a);
            }
            return cudaGetLastError();
        }
    }
    if (kind == 5) {  // tensor cores, BF16 storage only; one site per warp, N = 32 R
        if constexpr (std::is_same<S, bf16>::value && (R == 1 || R == 2)) {
            if (a.N != 32 * R) return cudaErrorInvalidValue;
            static size_t opted = 0;
            static std::mutex m;
            auto kern = hop_kernel_mma<R, MODE, RED>;
            l.block = WS_WARPS * 32;
            l.smem = MmaShape<R>::SMEM;
            const cudaError_t e = opt_in_smem(kern, l.smem, opted, m);
            if (e != cudaSuccess) return e;
            const int res = resident_blocks(kern, l.block, l.smem);
            l.grid = (l.num_sms > 0 ? l.num_sms : 1) * (res < 16 ? res : 16);
            kern<<<l.grid, l.block, l.smem, l.stream>>>(a);
            return cudaGetLastError();
        }
    }
    return cudaErrorInvalidValue;
}

// The (MODE, RED) combinations the solvers use, for storage type S and R
// right-hand sides per thread.  Each (S, R) pair is instantiated in its own
// translation unit (hop_f32.cu, hop_f32_r2.cu, ...), so the build compiles the
// kernel variants in parallel.
template <typename S, int R>
cudaError_t launch_hop_low_r(int mode, int red, int kind, const HopArgs &a, Launch &l) {
#define DL_CASE(m, rd) \
    if (mode == m && red == rd) return go_hop<S, R, m, rd>(a, l, kind);
    DL_CASE(MODE_PLAIN, RED_NONE)
    DL_CASE(MODE_XPAY, RED_NONE)
    DL_CASE(MODE_XPAY, RED_R0DOT)
    DL_CASE(MODE_XPAY, RED_BICG)
    DL_CASE(MODE_XPAY, RED_NORM)
#undef DL_CASE
    return cudaErrorInvalidValue;
}

// The R = 2 and R = 4 instantiations (hop_*_r2.cu, hop_*_r4.cu).
cudaError_t launch_hop_f32_r2(int mode, int red, int kind, const HopArgs &a, Launch &l);
cudaError_t launch_hop_f32_r4(int mode, int red, int kind, const HopArgs &a, Launch &l);
cudaError_t launch_hop_bf16_r2(int mode, int red, int kind, const HopArgs &a, Launch &l);
cudaError_t launch_hop_bf16_r4(int mode, int red, int kind, const HopArgs &a, Launch &l);

}  // namespace dl
