// Exchange of binary32 values between the blocks of a persistent launch through L2 (k_loop.cu,
// k_power.cu): 8-byte words of a value and a tag, which the reader polls, every wait
// bounded.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tvcs {

__device__ __forceinline__ int fresh_tid()   // not kept from one section to the next
{
    int t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}

// Tagged words: value in the low half, tag in the high half.
__device__ __forceinline__ uint64_t tagged(float v, uint32_t tag)
{
    return ((uint64_t)tag << 32) | __float_as_uint(v);
}

__device__ __forceinline__ void send2(uint64_t* p, float a, float b, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(tagged(a, tag)),
                 "l"(tagged(b, tag))
                 : "memory");
}

__device__ __forceinline__ ulonglong2 peek2(const uint64_t* p)
{
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ bool has_tag(ulonglong2 v, uint32_t tag)
{
    return (uint32_t)(v.x >> 32) == tag && (uint32_t)(v.y >> 32) == tag;
}

__device__ __forceinline__ float word_f(uint64_t v) { return __uint_as_float((uint32_t)v); }

// Bound of a block's waits, and its record that one gave up.
struct Waits {
    long long budget;
    volatile int* gave_up;   // shared memory
};

// The two words at p once both carry `tag` (v: a first look at them); whatever is there
// when the budget runs out or another wait of the block has given up.
__device__ __forceinline__ ulonglong2 await2(const uint64_t* p, uint32_t tag, ulonglong2 v, const Waits& w)
{
    if (has_tag(v, tag)) return v;
    const long long t0 = clock64();
    for (;;) {
        v = peek2(p);
        if (has_tag(v, tag)) return v;
        if (*w.gave_up) return v;
        if (clock64() - t0 > w.budget) {
            *w.gave_up = 1;
            return v;
        }
    }
}

// The two words at each of n <= K places of the exchange buffer once all carry `tag`;
// whatever is there when the budget runs out or another wait of the block has given up.
template <int K, class F>
__device__ __forceinline__ void poll2(ulonglong2* v, int n, uint32_t tag, const Waits& w, F at)
{
    long long t0 = 0;
    for (;;) {
        bool ok = true;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < n) v[k] = peek2(at(k));
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < n) ok = ok && has_tag(v[k], tag);
        if (ok || *w.gave_up) return;
        const long long t = clock64();
        if (t0 == 0) t0 = t;
        if (t - t0 > w.budget) {
            *w.gave_up = 1;
            return;
        }
    }
}

}  // namespace tvcs
