// What the single-pass products (k_products.cu) and the persistent iteration loop
// (k_loop.cu) share: how a block splits a row's columns and its rows over threads, and
// how entries of A are read from a stage of the shared-memory ring.
#pragma once

#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include "common.cuh"

namespace tvcs {

// TC column threads of V vectors of VW columns each (N = TC VW V), RL row lanes,
// RB rows per lane and step; a stage of the ring holds one step's RL RB rows.
template <int PREC, int TC, int VW, int V, int RL, int RB, int NST>
struct ProdShape {
    static constexpr int THREADS = TC * RL, WARPS = THREADS / 32, WPR = TC / 32;
    static constexpr int N = TC * VW * V, CPT = VW * V, RS = RL * RB;
    static constexpr int B0 = PREC == 0 ? 4 : PREC == 1 ? 2 : 1, B1 = PREC == 0 ? 0 : 2;   // bytes per entry
    static constexpr size_t P1_OFF = (size_t)RS * N * B0;          // second plane in a stage
    static constexpr size_t STAGE = (size_t)RS * N * (B0 + B1);
    static constexpr int YMAX = 1024;   // most rows of a block whose y (and scales) are fetched at its start
    static constexpr size_t O_BAR = NST * STAGE;
    static constexpr size_t O_RED = O_BAR + ((NST * 8 + 15) / 16) * 16;         // [2][RS][WPR]
    static constexpr size_t O_DRED = O_RED + ((2 * RS * WPR * 4 + 15) / 16) * 16;   // [32] float2
    static constexpr size_t O_FLAG = O_DRED + 32 * 8;
    static constexpr size_t O_Y = O_FLAG + 16;
    static constexpr size_t O_S = O_Y + YMAX * 4;
    static constexpr size_t SMEM = O_S + (PREC == 2 ? YMAX * 4 : 0);
    static_assert(TC % 32 == 0 && THREADS <= 512, "row lanes must be whole warps");
    static_assert((N * B0) % 16 == 0, "TMA sizes are multiples of 16 bytes");
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static_assert(2 * RS <= YMAX, "y of two steps");
    static_assert(NST * STAGE >= (size_t)(RL - 1) * N * 4 && NST * STAGE >= (size_t)WARPS * 32 * 16,
                  "the ring doubles as scratch of the epilogue");
};

__device__ __forceinline__ float lo16_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi16_f(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// BYTES of shared memory (4, 8 or 16, so aligned) as 32-bit words.
template <int BYTES>
__device__ __forceinline__ void lds_words(const unsigned char* p, uint32_t* w)
{
    static_assert(BYTES % 16 == 0 || BYTES == 8 || BYTES == 4 || BYTES == 2, "vector load");
    if constexpr (BYTES % 16 == 0) {
#pragma unroll
        for (int k = 0; k < BYTES / 16; ++k) {
            const uint4 v = reinterpret_cast<const uint4*>(p)[k];
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
    } else if constexpr (BYTES == 8) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x;
        w[1] = v.y;
    } else if constexpr (BYTES == 4) {
        w[0] = *reinterpret_cast<const uint32_t*>(p);
    } else {
        w[0] = *reinterpret_cast<const uint16_t*>(p);
    }
}

// VW consecutive entries of one row, starting at column c, as packed pairs of
// binary32: p0, p1 point at the row in the storage's planes, s is the row's scale (fp8).
template <int PREC, int VW>
__device__ __forceinline__ void load_entries(const unsigned char* p0, const unsigned char* p1, int c,
                                             float s, uint64_t* a)
{
    if constexpr (PREC == 0) {
        if constexpr (VW % 4 == 0) {
#pragma unroll
            for (int k = 0; k < VW / 4; ++k) {
                const ulonglong2 v = reinterpret_cast<const ulonglong2*>(p0 + (size_t)c * 4)[k];
                a[2 * k] = v.x;
                a[2 * k + 1] = v.y;
            }
        } else {
            a[0] = *reinterpret_cast<const uint64_t*>(p0 + (size_t)c * 4);
        }
    } else if constexpr (PREC == 1) {   // hi + lo, exact
        uint32_t h[VW / 2], l[VW / 2];
        lds_words<VW * 2>(p0 + (size_t)c * 2, h);
        lds_words<VW * 2>(p1 + (size_t)c * 2, l);
#pragma unroll
        for (int k = 0; k < VW / 2; ++k)
            a[k] = add2(pack2(lo16_f(h[k]), hi16_f(h[k])), pack2(lo16_f(l[k]), hi16_f(l[k])));
    } else {   // s q + c, one rounding
        uint32_t q[(VW + 3) / 4], cw[VW / 2];
        lds_words<VW>(p0 + c, q);
        lds_words<VW * 2>(p1 + (size_t)c * 2, cw);
        const uint64_t s2 = pack2(s, s);
#pragma unroll
        for (int k = 0; k < VW / 2; ++k) {
            const uint32_t pair = (q[k / 2] >> (16 * (k & 1))) & 0xffffu;
            const float2 f = __half22float2(
                __half2(__nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)pair, __NV_E4M3)));
            a[k] = fma2(s2, pack2(f.x, f.y), pack2(lo16_f(cw[k]), hi16_f(cw[k])));
        }
    }
}

}  // namespace tvcs
