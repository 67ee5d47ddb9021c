// The power iteration of a handle up to 64 x 64 whose rows of A all fit on chip (v <- A^T A v /
// ||A^T A v||, from which tau is taken), all rounds in one persistent cooperative launch.
//
// G blocks, one per SM, each with a contiguous range of rows of A for the whole launch, as
// binary32: RL RREG of them in registers, the rest in shared memory.  Every block keeps the whole
// v, so that only A^T r travels, as the words of loop_exchange.cuh: with few blocks every block
// adds all partials, else the owner of a slice of SL columns adds its partials and sends the
// sums to all, with its part of ||g||^2 (binary64 runs at 1/64 of the binary32 rate here: every
// block squaring all of g took 2 of 10 us a round at 64 x 64).  A buffer is written again only after every block has sent something that it could
// not have sent before reading the buffer.
//
// What bounds it: latency (one or two exchanges of about 1.2 us and six block barriers a round;
// the products are 0.5 us).  A launch of the products, one of the partials' sum and one of the
// scaling took about 20 us a round at every size; tvcs_create with 100 rounds: 16 x 16 (m = 77)
// 1.87 -> 0.49 ms, 32 x 32 (307) 2.49 -> 0.93, 48 x 48 (691) 2.74 -> 1.08, 64 x 64 (1229) 3.12 -> 1.44.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "loop_exchange.cuh"
#include "loop_rows.cuh"

namespace tvcs {

namespace {

struct PowerState {
    int gave_up;            // a wait ran out
    int last;               // this block is the last to end
    float s1, s2, hi, lo;   // 1 / ||g|| = s1 s2 (hi + lo), s1 and s2 powers of two
};

template <int NN_, int TC_, int V_, int RL_, int RREG_>
struct PowerShape {
    static constexpr int NN = NN_, TC = TC_, V = V_, RL = RL_, RREG = RREG_, SL = 32;
    static constexpr int N = NN * NN, THREADS = TC * RL, WPR = TC / 32, CP = 2 * V;
    static_assert(TC * V * 4 == N && TC % 32 == 0 && RREG % 4 == 0 && THREADS <= 512, "split");
    static constexpr int GRP = THREADS / (SL / 2);          // groups of partials in a slice's sums
    static_assert(N % SL == 0 && THREADS % (SL / 2) == 0 && GRP % 2 == 0, "slices");
    static constexpr int RROWS = RL * RREG;                 // rows in registers
    static constexpr int RED = WPR | 1;                     // stride of a row's warp sums (odd banks)
    static constexpr size_t al(size_t b) { return (b + 15) / 16 * 16; }
    static constexpr size_t O_V = 0;
    static constexpr size_t O_STATE = O_V + N * 4;
    static constexpr size_t O_DRED = O_STATE + al(sizeof(PowerState));   // [32] of 8 bytes
    static constexpr size_t O_SCR = O_DRED + 32 * 8;                     // the lanes', the groups' sums
    static constexpr size_t SCR = al(std::max(RL > 1 ? (size_t)RL * N * 4 : 0, (size_t)GRP * SL * 4));
    static constexpr size_t O_RED = O_SCR + SCR;
    static constexpr size_t ROW_BYTES = (size_t)RED * 4 + 4;             // a row's warp sums and r
    static constexpr size_t LIMIT = 227 * 1024;
    // rows in shared memory besides the RROWS in registers
    static constexpr int XMAX = (int)((LIMIT - O_RED - 64 - RROWS * ROW_BYTES) / ((size_t)N * 4 + ROW_BYTES));
    static constexpr int RMAX = RROWS + XMAX;
    static constexpr size_t O_R = al(O_RED + (size_t)RMAX * RED * 4);
    static constexpr size_t O_A = al(O_R + (size_t)RMAX * 4);
    static constexpr size_t smem(int rows) { return O_A + (size_t)std::max(0, rows - RROWS) * N * 4; }
    static_assert(smem(RMAX) <= LIMIT, "shared memory");
};

#define POWER_SMEM extern __shared__ __align__(128) unsigned char smem[]
#define POWER_AT(T, off) reinterpret_cast<T*>(smem + (off))

// 1 / sqrt(s) = st->s1 st->s2 (st->hi + st->lo); NaN where sqrt(s) is 0 or not finite.
__device__ __forceinline__ void power_inverse_norm(PowerState* st, double s)
{
    const double nrm = sqrt(s);
    const bool ok = nrm > 0.0 && isfinite(nrm);
    const int e = ok ? ilogb(nrm) : 0;   // |e| <= 160 for sums of binary32 squares
    const double f = ok ? 1.0 / ldexp(nrm, -e) : nan("");
    st->s1 = ldexpf(1.f, -(e / 2));
    st->s2 = ldexpf(1.f, -(e - e / 2));
    st->hi = (float)f;
    st->lo = (float)(f - (double)st->hi);
}

// v <- v / ||v||, the sum of the threads' s being ||v||^2 in binary64 (it may be out of binary32's
// range).  The quotient is v (hi + lo) by one product and one FMA in binary32, within an ulp of the
// binary64 division's (which the chain of launches uses): the error of tau, mean of eight inputs, is
// 6.8, 9.2, 5.5, 2.3e-9 at n = 16, 32, 48, 64 (with the division 8.8, 8.2, 6.3, 4.6e-9).
template <class S>
__device__ __forceinline__ void power_normalize(double s)
{
    POWER_SMEM;
    const int tid = fresh_tid();
    PowerState* st = POWER_AT(PowerState, S::O_STATE);
    float* sv = POWER_AT(float, S::O_V);
    s = block_sum(s, POWER_AT(double, S::O_DRED));
    if (tid == 0) power_inverse_norm(st, s);
    __syncthreads();
    const float s1 = st->s1, s2 = st->s2, hi = st->hi, lo = st->lo;
    for (int i = tid; i < S::N; i += S::THREADS) {
        const float z = sv[i] * s1 * s2;
        sv[i] = fmaf(z, hi, z * lo);
    }
    __syncthreads();
}

}  // namespace

template <int NN, int TC, int V, int RL, int RREG>
__global__ void __launch_bounds__(TC * RL, 1) k_power(const __grid_constant__ PowerArgs q)
{
    using S = PowerShape<NN, TC, V, RL, RREG>;
    constexpr int N = S::N, T = S::THREADS, CP = S::CP, RROWS = S::RROWS, GRP = S::GRP, SL = S::SL;
    POWER_SMEM;
    const int tid = threadIdx.x, lane = tid & 31;
    const int lane_row = tid / TC, ltid = tid - lane_row * TC;
    const int G = gridDim.x, blk = blockIdx.x;
    float* sv = POWER_AT(float, S::O_V);
    float* scr = POWER_AT(float, S::O_SCR);
    float* sr = POWER_AT(float, S::O_R);
    float* srow = POWER_AT(float, S::O_A);
    PowerState* st = POWER_AT(PowerState, S::O_STATE);
    const int i0 = (int)(((long long)q.m * blk) / G);
    const int nrows = (int)(((long long)q.m * (blk + 1)) / G) - i0;
    const Waits waits{q.budget, &st->gave_up};
    uint64_t a[RREG][CP];
    reg_load_rows<S>(q, i0, nrows, lane_row, ltid, a, srow);
    for (int i = tid; i < N; i += T) sv[i] = q.v0;
    if (tid == 0) st->gave_up = 0;
    __syncthreads();

    const bool two = G > q.one_max;   // two exchanges
    for (int it = 1;; ++it) {         // `iters` rounds, then a last pass for ||A v||
        const uint32_t tag = q.tag0 + (uint32_t)it;
        uint64_t x[CP], acc[CP];
        reg_cols<S>(sv, ltid, x);
        reg_residual<S>(a, x, srow, nullptr, POWER_AT(float, S::O_RED), sr, nrows, tid);
        if (it > q.iters) break;
        reg_adjoint<S>(a, srow, sr, nrows, lane_row, ltid, acc);

        // the partial, two exchanges: [slice][block][SL], one: [round & 1][block][N]
        uint64_t* part = q.xbuf + (two ? 0 : (size_t)(it & 1) * G * N);
        uint64_t* sums = q.xbuf + (size_t)G * N;   // two exchanges: the sums, then every slice's part of ||g||^2
        uint64_t* norms = sums + N;
        double sq = 0.0;
        auto send_partial = [&](int c, uint64_t pair) {
            const float2 t = unpack2(pair);
            send2(two ? part + ((size_t)(c / SL) * G + blk) * SL + c % SL : part + (size_t)blk * N + c, t.x, t.y, tag);
        };
        auto lanes_sum = [&](int i) {   // columns 2 i, 2 i + 1 over the row lanes
            uint64_t s = reinterpret_cast<const uint64_t*>(scr)[i];
#pragma unroll
            for (int l = 1; l < RL; ++l) s = add2(s, reinterpret_cast<const uint64_t*>(scr)[l * (N / 2) + i]);
            return s;
        };
        if constexpr (RL > 1) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                *reinterpret_cast<ulonglong2*>(scr + (size_t)lane_row * N + (ltid + v * TC) * 4) =
                    make_ulonglong2(acc[2 * v], acc[2 * v + 1]);
            __syncthreads();
            if (G > 1)
                for (int i = tid; i < N / 2; i += T) send_partial(2 * i, lanes_sum(i));
        } else {
#pragma unroll
            for (int c = 0; c < CP; ++c) send_partial((ltid + (c / 2) * TC) * 4 + 2 * (c % 2), acc[c]);
        }
        if (two) {   // a slice's owner adds its partials and sends the sums
            if constexpr (RL > 1) __syncthreads();   // (the lanes' sums are read)
#pragma unroll 1
            for (int s = blk; s < N / SL; s += G) {
                const int pair = tid % (SL / 2), grp = tid / (SL / 2);
                const uint64_t* src = part + ((size_t)s * G + grp) * SL + 2 * pair;
                float2 t = make_float2(0.f, 0.f);
                constexpr int K = 152 / GRP + 1;   // one batch on 152 SMs
#pragma unroll 1
                for (int b = grp; b < G; b += GRP * K, src += (size_t)GRP * K * SL) {
                    ulonglong2 v[K];
                    const int n = min(K, (G - b + GRP - 1) / GRP);
                    poll2<K>(v, n, tag, waits, [&](int k) { return src + (size_t)k * GRP * SL; });
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (k < n) {
                            t.x += word_f(v[k].x);
                            t.y += word_f(v[k].y);
                        }
                }
                if (s != blk) __syncthreads();   // (the previous slice's sums are read)
                reinterpret_cast<float2*>(scr)[grp * (SL / 2) + pair] = t;
                __syncthreads();
                if (tid < 32) {
                    float2 z = make_float2(0.f, 0.f);
                    const int c = lane & 15, h = lane >> 4;
#pragma unroll
                    for (int g = 0; g < GRP / 2; ++g) {
                        const float2 e = reinterpret_cast<const float2*>(scr)[(h * (GRP / 2) + g) * (SL / 2) + c];
                        z.x += e.x;
                        z.y += e.y;
                    }
                    z.x += __shfl_xor_sync(0xffffffffu, z.x, 16);
                    z.y += __shfl_xor_sync(0xffffffffu, z.y, 16);
                    if (h == 0) send2(sums + (size_t)s * SL + 2 * c, z.x, z.y, tag);
                    double d = fma((double)z.y, (double)z.y, (double)z.x * (double)z.x);
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                    if (lane == 0)
                        send2(norms + 2 * s, __int_as_float(__double2loint(d)), __int_as_float(__double2hiint(d)), tag);
                }
            }
            constexpr int K = (N / 2 + T - 1) / T;
            ulonglong2 v[K];
            const int n = (N / 2 - tid + T - 1) / T;
            poll2<K>(v, n, tag, waits, [&](int k) { return sums + 2 * (tid + k * T); });
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < n) reinterpret_cast<float2*>(sv)[tid + k * T] = make_float2(word_f(v[k].x), word_f(v[k].y));
            static_assert(N / SL <= T, "a slice's norm a thread");
            if (tid < N / SL) {
                ulonglong2 d[1];
                poll2<1>(d, 1, tag, waits, [&](int) { return norms + 2 * tid; });
                sq = __hiloint2double((int)(uint32_t)d[0].y, (int)(uint32_t)d[0].x);
            }
        } else if (G > 1) {
#pragma unroll 1
            for (int i = tid; i < N / 2; i += T) {
                const uint64_t* src = part + 2 * i;
                float2 t = make_float2(0.f, 0.f);
                constexpr int K = 8;
#pragma unroll 1
                for (int b = 0; b < G; b += K, src += (size_t)K * N) {
                    ulonglong2 v[K];
                    const int n = min(K, G - b);
                    poll2<K>(v, n, tag, waits, [&](int k) { return src + (size_t)k * N; });
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (k < n) {
                            t.x += word_f(v[k].x);
                            t.y += word_f(v[k].y);
                        }
                }
                reinterpret_cast<float2*>(sv)[i] = t;
            }
        } else if constexpr (RL > 1) {   // one block
            for (int i = tid; i < N / 2; i += T) reinterpret_cast<uint64_t*>(sv)[i] = lanes_sum(i);
        }
        // (the vote makes the outcome the same for every thread of the block)
        if (__syncthreads_or(st->gave_up)) break;
        if (!two)
            for (int i = tid; i < N; i += T) sq = fma((double)sv[i], (double)sv[i], sq);
        power_normalize<S>(sq);
    }

    // ||A v||^2 over the blocks, by the last one to come
    float2 r2 = make_float2(0.f, 0.f);
    for (int i = tid; i < nrows; i += T) r2 = ds_add(r2, ds_sq(sr[i]));
    r2 = block_sum_ds(r2, POWER_AT(float2, S::O_DRED));
    if (tid == 0) {
        if (st->gave_up) set_error(q.ctrl, ERR_TIMEOUT);
        q.r2part[blk] = r2;
    }
    if (!last_block_all(&q.ctrl->ticket_gather, &st->last)) return;
    float2 v = make_float2(0.f, 0.f);
    for (int b = tid; b < G; b += T) v = ds_add(v, __ldcg(q.r2part + b));
    v = block_sum_ds(v, POWER_AT(float2, S::O_DRED));
    if (tid == 0) q.ctrl->r2 = ds_value(v);
}

// ---------------------------------------------------------------------------
// Shapes: n -> (rows per block aimed at, most blocks with one exchange, TC, V, RL, RREG).
// ---------------------------------------------------------------------------
#define TVCS_POWER_TABLE(X)           \
    X(16, 256, 32, 32, 2, 8, 16)      \
    X(32, 32, 16, 128, 2, 2, 16)      \
    X(48, 8, 16, 192, 3, 2, 4)        \
    X(64, 8, 16, 256, 4, 1, 8)

template <int NN, int TC, int V, int RL, int RREG>
static bool power_configure_t()
{
    using S = PowerShape<NN, TC, V, RL, RREG>;
    auto kernel = k_power<NN, TC, V, RL, RREG>;
    int per = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem(S::RMAX)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, S::THREADS, S::smem(S::RMAX)) != cudaSuccess ||
        per < 1) {
        cudaGetLastError();
        return false;
    }
    return true;
}

bool power_configure(int n)
{
#define X(NN, TGT, ONE, TC, V, RL, RREG) \
    if (n == NN) return power_configure_t<NN, TC, V, RL, RREG>();
    TVCS_POWER_TABLE(X)
#undef X
    return false;
}

int power_grid(int n, int m, int num_sms)
{
#define X(NN, TGT, ONE, TC, V, RL, RREG)                                                                   \
    if (n == NN) {                                                                                         \
        const int g = std::max(RL > 1 ? 1 : 2, std::min(num_sms, (m + TGT - 1) / TGT));                    \
        return g <= num_sms && (m + g - 1) / g <= PowerShape<NN, TC, V, RL, RREG>::RMAX ? g : 0;           \
    }
    TVCS_POWER_TABLE(X)
#undef X
    return 0;
}

size_t power_words(int n, int grid)
{
    const size_t N = (size_t)n * n;
    int one = 0;
#define X(NN, TGT, ONE, TC, V, RL, RREG) \
    if (n == NN) one = ONE;
    TVCS_POWER_TABLE(X)
#undef X
    // one exchange: two sets of partials; two: one set, the sums, two words of norm a slice
    return grid <= one ? 2 * grid * N : (grid + 1) * N + 2 * (N / 32);
}

cudaError_t launch_power(int n, int grid, PowerArgs a, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // the blocks wait for one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define X(NN, TGT, ONE, TC, V, RL, RREG)                                 \
    if (n == NN) {                                                       \
        using S = PowerShape<NN, TC, V, RL, RREG>;                       \
        a.one_max = ONE;                                                 \
        cfg.blockDim = dim3(S::THREADS, 1, 1);                           \
        cfg.dynamicSmemBytes = S::smem((a.m + grid - 1) / grid);         \
        return cudaLaunchKernelEx(&cfg, k_power<NN, TC, V, RL, RREG>, a);\
    }
    TVCS_POWER_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace tvcs
