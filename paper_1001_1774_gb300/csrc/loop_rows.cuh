// What the loop kernels that keep every row of A on chip share (k_loop.cu, k_power.cu): a
// thread has V vectors of 4 columns, TC of them apart, of RREG rows in registers, as binary32.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "products.cuh"

namespace tvcs {

// Sums of four values over the lanes of a warp in 6 shuffles: afterwards lane l holds the sum
// of value 2 (l & 1) + (l >> 1 & 1).
__device__ __forceinline__ float warp_sum4(const float* v, int lane)
{
    const bool b0 = lane & 1, b1 = lane & 2;
    float p = (b0 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b0 ? v[0] : v[2], 1);
    float q = (b0 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, b0 ? v[1] : v[3], 1);
    float s = (b1 ? q : p) + __shfl_xor_sync(0xffffffffu, b1 ? p : q, 2);
#pragma unroll
    for (int o = 4; o < 32; o *= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// The thread's columns of a row in shared memory.
template <class S>
__device__ __forceinline__ void reg_cols(const float* row, int ltid, uint64_t* e)
{
#pragma unroll
    for (int v = 0; v < S::V; ++v) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(row + (ltid + v * S::TC) * 4);
        e[2 * v] = t.x;
        e[2 * v + 1] = t.y;
    }
}

template <class S>
__device__ __forceinline__ float reg_dot(const uint64_t* a, const uint64_t* x)
{
    uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
    for (int c = 0; c < S::CP; c += 2) {
        s0 = fma2(a[c], x[c], s0);
        s1 = fma2(a[c + 1], x[c + 1], s1);
    }
    const float2 t = unpack2(add2(s0, s1));
    return t.x + t.y;
}

// The thread's columns of row `row` of A, decoded.  (Q: P0, P1, rscale, prec.)
template <class S, class Q>
__device__ __forceinline__ void reg_load_row(const Q& q, int row, int ltid, uint64_t* e)
{
    const size_t o = (size_t)row * S::N;
#pragma unroll
    for (int v = 0; v < S::V; ++v) {
        const int c = (ltid + v * S::TC) * 4;
        if (q.prec == 0)
            load_entries<0, 4>(q.P0 + o * 4, nullptr, c, 1.f, e + 2 * v);
        else if (q.prec == 1)
            load_entries<1, 4>(q.P0 + o * 2, q.P1 + o * 2, c, 1.f, e + 2 * v);
        else
            load_entries<2, 4>(q.P0 + o, q.P1 + o * 2, c, q.rscale[row], e + 2 * v);
    }
}

// The block's rows i0 .. i0 + nrows - 1 of A: row lane_row RREG + b to registers, those past
// S::RROWS to shared memory.
template <class S, class Q>
__device__ __forceinline__ void reg_load_rows(const Q& q, int i0, int nrows, int lane_row, int ltid,
                                              uint64_t (&a)[S::RREG][S::CP], float* srow)
{
#pragma unroll
    for (int b = 0; b < S::RREG; ++b) {
        const int row = lane_row * S::RREG + b;
#pragma unroll
        for (int c = 0; c < S::CP; ++c) a[b][c] = 0ull;
        if (row < nrows) reg_load_row<S>(q, i0 + row, ltid, a[b]);
    }
    for (int x = lane_row; x < nrows - S::RROWS; x += S::RL) {
        uint64_t e[S::CP];
        reg_load_row<S>(q, i0 + S::RROWS + x, ltid, e);
#pragma unroll
        for (int v = 0; v < S::V; ++v)
            *reinterpret_cast<ulonglong2*>(srow + (size_t)x * S::N + (ltid + v * S::TC) * 4) =
                make_ulonglong2(e[2 * v], e[2 * v + 1]);
    }
}

// r = A x - f of the block's rows (f: shared memory, or null for 0), into sr; two block barriers.
// red: scratch for the warps' sums, S::RED a row.
template <class S>
__device__ __forceinline__ void reg_residual(const uint64_t (&a)[S::RREG][S::CP], const uint64_t* x, const float* srow,
                                             const float* f, float* red, float* sr, int nrows, int tid)
{
    constexpr int RL = S::RL, CP = S::CP, WPR = S::WPR, RREG = S::RREG, RROWS = S::RROWS;
    const int lane = tid & 31, lane_row = tid / S::TC, ltid = tid - lane_row * S::TC, xr = nrows - RROWS;
    const int k4 = 2 * (lane & 1) + (lane >> 1);   // whose sum lane 0..3 holds after warp_sum4
#pragma unroll
    for (int b = 0; b < RREG; b += 4) {
        float d[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = reg_dot<S>(a[b + k], x);
        const float s = warp_sum4(d, lane);
        if (lane < 4) red[(lane_row * RREG + b + k4) * S::RED + (ltid >> 5)] = s;
    }
#pragma unroll 1
    for (int x0 = 4 * lane_row; x0 < xr; x0 += 4 * RL) {
        float d[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            d[k] = 0.f;
            if (x0 + k < xr) {
                uint64_t e[CP];
                reg_cols<S>(srow + (size_t)(x0 + k) * S::N, ltid, e);
                d[k] = reg_dot<S>(e, x);
            }
        }
        const float s = warp_sum4(d, lane);
        if (lane < 4 && x0 + k4 < xr) red[(RROWS + x0 + k4) * S::RED + (ltid >> 5)] = s;
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < nrows; i += S::THREADS) {
        float t[WPR];
#pragma unroll
        for (int w = 0; w < WPR; ++w) t[w] = red[i * S::RED + w];
#pragma unroll
        for (int o = 1; o < WPR; o *= 2)
#pragma unroll
            for (int w = 0; w + o < WPR; w += 2 * o) t[w] += t[w + o];
        sr[i] = f ? t[0] - f[i] : t[0];
    }
    __syncthreads();
}

// The row lane's part of A^T r: the thread's columns.
template <class S>
__device__ __forceinline__ void reg_adjoint(const uint64_t (&a)[S::RREG][S::CP], const float* srow, const float* sr,
                                            int nrows, int lane_row, int ltid, uint64_t* acc)
{
    constexpr int CP = S::CP;
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0ull;
#pragma unroll
    for (int b = 0; b < S::RREG; ++b) {
        const int row = lane_row * S::RREG + b;
        const float ri = row < nrows ? sr[row] : 0.f;
        const uint64_t rr = pack2(ri, ri);
#pragma unroll
        for (int c = 0; c < CP; ++c) acc[c] = fma2(rr, a[b][c], acc[c]);
    }
#pragma unroll 2
    for (int x = lane_row; x < nrows - S::RROWS; x += S::RL) {
        const float ri = sr[S::RROWS + x];
        const uint64_t rr = pack2(ri, ri);
        uint64_t e[CP];
        reg_cols<S>(srow + (size_t)x * S::N, ltid, e);
#pragma unroll
        for (int c = 0; c < CP; ++c) acc[c] = fma2(rr, e[c], acc[c]);
    }
}

}  // namespace tvcs
