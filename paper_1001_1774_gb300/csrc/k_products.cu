// Rows a6-a7: r = A x - y and g = A^T r in ONE pass over A (Xiao & Yang,
// eq. (line): g_k = A^T (A u^k - f); two products per iteration, Sec. 3.1), for
// images up to 128 x 128 and every storage of A (k_products_q.cu has the larger
// ones and states the storages: binary32, bf16 hi + lo, fp8 e4m3 + bf16).
//
// Each block owns a contiguous range of rows of A.  Thread 0 streams them into
// a ring of NST stages of RS rows in shared memory with bulk asynchronous copies
// (TMA, non-tensor form, one mbarrier per stage; A is read once per call, with
// an L2 evict-first hint), the first stages before the dependency wait on the
// preceding kernel, together with an L2 prefetch of the block's next rows.  A
// thread owns fixed columns: it reads its columns of RB rows into registers
// (decoded to binary32 once), forms the dot products with x (warp shuffles + one
// named barrier for all RB rows), computes r_i = dot - y_i and folds r_i A_i into
// its accumulators of A^T r from the same registers.  Each block writes its
// partial A^T r (N floats); with g_out set, a grid barrier (cooperative launch)
// follows and every block sums its slice of the P partials in a fixed order
// (deterministic), otherwise a later kernel does.
//
// What bounds it: HBM, once a row's step (stage wait, loads, warp shuffles, block
// barrier, update; all warps in step) does not.  A row crosses shared memory twice
// (written by the copy, read once) and is multiplied by packed FMAs (two columns an
// instruction): at n = 128 a step takes about 1,250 cycles when its 64 KB are there,
// against about 2,050 when the row was read again from shared memory for A^T r with
// scalar FMAs, which held an iteration at 55.0 us whatever was prefetched (52.1 now;
// bf16 hi + lo 70.1 -> 54.9, fp8 + bf16 61.2 -> 46.8, whose launches also had no
// overlap with the u-solve and a separate reduction kernel; n = 96, m = 2765:
// 25.0 -> 23.7).  The named barrier also frees the stage (every thread has its
// columns in registers when it arrives), so no second mbarrier is needed.  RB rows
// share one barrier where the columns per thread leave registers for them.
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "products.cuh"

namespace tvcs {

// Rows of A prefetched into L2 per block before the dependency wait, beyond the
// ring: 1 MB (16 rows at n = 128; 136 blocks then hold about L2's capacity).
constexpr size_t PROD_PF_BYTES = 1024 * 1024;

// One block per SM (the ring fills shared memory at the larger sizes); the grid
// leaves 16 SMs to the u-solve cluster of the same iteration, which runs there
// while this kernel streams A.
//
// BIG: a block may have more than YMAX rows.  Up to that many, y (and the scales) of a block's
// rows are fetched into shared memory at the start, so that no step waits on a global load
// for them.  BIG: one thread a row fetches y with each step, into two sets of a step's rows, and
// before the step's barrier: r may be stored over y (tvcs_apply_noalloc), so nobody may look for y
// after it.  (Two kernels, because one that chose inside the step cost n = 128 up to 1 %: us an
// iteration, binary32 52.0, bf16 56.4, fp8 48.1 where it read y of such blocks after the barrier,
// 52.1, 56.3, 47.7 with the choice, 52.0, 56.0, 45.7 as two.)
template <int PREC, int TC, int VW, int V, int RL, int RB, int NST, bool BIG>
__global__ void __maxnreg__(128)
    k_products(const unsigned char* __restrict__ P0, const unsigned char* __restrict__ P1,
               const float* __restrict__ rscale, int m, const float* __restrict__ x,
               const float* __restrict__ y, float* __restrict__ r, float* __restrict__ gpart,
               float* __restrict__ g_out, float2* __restrict__ r2part, Ctrl* __restrict__ ctrl,
               int mode, cudaGraphConditionalHandle cond, int set_cond, long long budget, int pf,
               int bar_extra, int* host_err)
{
    using S = ProdShape<PREC, TC, VW, V, RL, RB, NST>;
    constexpr int N = S::N, WPR = S::WPR, RS = S::RS, CPT = S::CPT, THREADS = S::THREADS;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::O_BAR);
    float* red = reinterpret_cast<float*>(smem + S::O_RED);
    float2* dred = reinterpret_cast<float2*>(smem + S::O_DRED);
    int* sflag = reinterpret_cast<int*>(smem + S::O_FLAG);
    float* sy = reinterpret_cast<float*>(smem + S::O_Y);
    float* ss = reinterpret_cast<float*>(smem + S::O_S);

    const int tid = threadIdx.x;
    const int G = gridDim.x;
    const int i0 = (int)(((long long)m * blockIdx.x) / G);
    const int i1 = (int)(((long long)m * (blockIdx.x + 1)) / G);
    const int nrows = i1 - i0;
    const int nst = (nrows + RS - 1) / RS;

    if (tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(&full[s], 1);
        fence_mbar_init();
    }
    __syncthreads();

    // The TMA copies are issued by thread 0.  A does not depend on the preceding
    // kernel: the first NST stages go out before the dependency wait, so
    // that under a programmatic dependent launch they stream in while the
    // u-solve still runs.
    const uint64_t pol = l2_policy_evict_first();
    auto issue = [&](int s) {
        const int slot = s % NST;
        const int b0 = s * RS;
        const size_t row = (size_t)(i0 + b0);
        const uint32_t ent = (uint32_t)min(RS, nrows - b0) * N;
        unsigned char* dst = smem + (size_t)slot * S::STAGE;
        mbar_arrive_expect_tx(&full[slot], ent * (S::B0 + S::B1));
        tma_load_1d(dst, P0 + row * N * S::B0, ent * S::B0, &full[slot], pol);
        if constexpr (S::B1 > 0)
            tma_load_1d(dst + S::P1_OFF, P1 + row * N * S::B1, ent * S::B1, &full[slot], pol);
    };
    // The pf stages after the ring are prefetched into L2 before the wait as
    // well (nothing waits for them): while the u-solve still runs, HBM streams
    // more of A than the ring holds, and the ring's later copies find those
    // rows in L2.  (Prefetching further ahead during the stream measured slower.)
    auto prefetch = [&](int s) {
        const int b0 = s * RS;
        const size_t row = (size_t)(i0 + b0);
        const uint32_t ent = (uint32_t)min(RS, nrows - b0) * N;
        prefetch_l2_bulk(P0 + row * N * S::B0, ent * S::B0);
        if constexpr (S::B1 > 0) prefetch_l2_bulk(P1 + row * N * S::B1, ent * S::B1);
    };
    const int pre = min(NST, nst);
    int issued = 0;   // stages issued (thread 0)
    if (tid == 0) {
        for (; issued < pre; ++issued) issue(issued);
        for (int s = pre; s < min(pre + pf, nst); ++s) prefetch(s);
    }
    pdl_wait();   // x and the control block come from the preceding u-solve
    if (mode == MODE_ITER) {
        const int skip = ctrl->skip;
        // The next u-solve writes skip before its own wait: release it only now.
        pdl_release();
        if (blockIdx.x == 0 && tid == 0) {
            if (!skip && ctrl->algo == 0) ctrl->pending = 1;
            if (set_cond) {
                // The loop ends when the run is done; `loops` bounds it independently.
                const int lc = ++ctrl->loops;
                const int cont =
                    (!ctrl->done && ctrl->error == ERR_NONE && lc < ctrl->loops_max) ? 1 : 0;
                cudaGraphSetConditional(cond, (unsigned)cont);
            }
        }
        if (skip) {   // leave no copy in flight
            if (tid == 0)
                for (int s = 0; s < pre; ++s) mbar_wait(&full[s], 0u, drain_budget(budget));
            return;
        }
    } else {
        pdl_release();
    }

    // ---------------- consumers ----------------
    if constexpr (!BIG) {
        for (int i = tid; i < nrows; i += THREADS) sy[i] = y != nullptr ? y[i0 + i] : 0.f;
        if constexpr (PREC == 2)
            for (int i = tid; i < nrows; i += THREADS) ss[i] = rscale[i0 + i];
    }
    const int lane_row = tid / TC;
    const int ltid = tid - lane_row * TC;
    const int warp_in_row = ltid >> 5;
    constexpr int CP = CPT / 2, VP = VW / 2;   // packed pairs of columns
    uint64_t xu[CP], acc[CP];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float* xv = x + (ltid + v * TC) * VW;
        if constexpr (VW % 4 == 0) {
#pragma unroll
            for (int k = 0; k < VW / 4; ++k) {
                const ulonglong2 t = reinterpret_cast<const ulonglong2*>(xv)[k];
                xu[v * VP + 2 * k] = t.x;
                xu[v * VP + 2 * k + 1] = t.y;
            }
        } else {
            xu[v] = *reinterpret_cast<const uint64_t*>(xv);
        }
    }
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0ull;
    named_barrier(1, THREADS);   // y and the scales are in shared memory
    float2 r2 = make_float2(0.f, 0.f);   // double-single ||r||^2 of this lane's rows (ltid == 0)
    bool ok = true;
    // After a wait gave up, the steps go on with what is in shared memory (every thread
    // stays with the block's barriers); the error word says that the results are void.
    for (int s = 0; s < nst; ++s) {
        const int slot = s % NST;
        if (ok && !mbar_wait(&full[slot], (s / NST) & 1, budget)) {
            set_error(ctrl, ERR_TIMEOUT, host_err);
            ok = false;
        }
        const unsigned char* sb = smem + (size_t)slot * S::STAGE;
        const int li0 = s * RS + lane_row * RB;   // first row of this lane's step, in the block
        uint64_t a[RB][CP];
        float* rb = red + ((s & 1) * RS + lane_row * RB) * WPR;
        [[maybe_unused]] float* yb = sy + (s & 1) * RS + lane_row * RB;
        float d[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            if (RS == 1 || li0 + b < nrows) {
                const size_t row = (size_t)(lane_row * RB + b) * N;
                float sc = 1.f;
                if constexpr (PREC == 2) sc = BIG ? rscale[i0 + li0 + b] : ss[li0 + b];
#pragma unroll
                for (int v = 0; v < V; ++v)
                    load_entries<PREC, VW>(sb + row * S::B0, sb + S::P1_OFF + row * S::B1,
                                           (ltid + v * TC) * VW, sc, &a[b][v * VP]);
            } else {
#pragma unroll
                for (int c = 0; c < CP; ++c) a[b][c] = 0ull;
            }
            uint64_t d0 = 0ull, d1 = 0ull;
#pragma unroll
            for (int c = 0; c < CP; ++c) {
                if (c & 1)
                    d1 = fma2(a[b][c], xu[c], d1);
                else
                    d0 = fma2(a[b][c], xu[c], d0);
            }
            const float2 t = unpack2(add2(d0, d1));
            d[b] = t.x + t.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int b = 0; b < RB; ++b) d[b] += __shfl_xor_sync(0xffffffffu, d[b], o);
        if ((tid & 31) == 0) {
#pragma unroll
            for (int b = 0; b < RB; ++b) rb[b * WPR + warp_in_row] = d[b];
        }
        if constexpr (BIG) {
            if (ltid == 0)
                for (int b = 0; b < RB; ++b)
                    if (li0 + b < nrows) yb[b] = y != nullptr ? y[i0 + li0 + b] : 0.f;
        }
        named_barrier(1, THREADS);   // the warps' parts are there, and nobody reads the stage any more
        // refill this slot with stage s + NST
        if (tid == 0 && ok && s + NST < nst) {
            issue(s + NST);
            ++issued;
        }
#pragma unroll
        for (int b = 0; b < RB; ++b) {
            const int li = li0 + b;
            if (RS > 1 && li >= nrows) break;
            float dot;
            if constexpr (WPR % 4 == 0) {   // fixed tree over the warps' parts
                uint64_t p[WPR / 2];
#pragma unroll
                for (int w = 0; w < WPR / 4; ++w) {
                    const ulonglong2 t = reinterpret_cast<const ulonglong2*>(rb + b * WPR)[w];
                    p[2 * w] = t.x;
                    p[2 * w + 1] = t.y;
                }
#pragma unroll
                for (int o = 1; o < WPR / 2; o *= 2)
#pragma unroll
                    for (int w = 0; w + o < WPR / 2; w += 2 * o) p[w] = add2(p[w], p[w + o]);
                const float2 t = unpack2(p[0]);
                dot = t.x + t.y;
            } else {
                dot = rb[b * WPR];
#pragma unroll
                for (int w = 1; w < WPR; ++w) dot += rb[b * WPR + w];
            }
            const float ri = dot - (BIG ? yb[b] : sy[li]);
            if (ltid == 0) {
                r[i0 + li] = ri;
                r2 = ds_add(r2, ds_sq(ri));
            }
            const uint64_t rr = pack2(ri, ri);
#pragma unroll
            for (int c = 0; c < CP; ++c) acc[c] = fma2(rr, a[b][c], acc[c]);
        }
    }
    if (tid == 0 && !ok)   // a wait gave up: let the copies still in flight land (bounded)
        for (int s = max(0, issued - NST); s < issued; ++s)
            mbar_wait(&full[s % NST], (s / NST) & 1, drain_budget(budget));

    // ---------------- epilogue: partial A^T r and ||r||^2 ----------------
    named_barrier(1, THREADS);   // every consumer is done with the stage ring
    float* out = gpart + (size_t)blockIdx.x * N;
    float* scr = reinterpret_cast<float*>(smem);   // (RL-1) x N
    if constexpr (RL > 1) {
        if (lane_row > 0) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                *reinterpret_cast<uint64_t*>(scr + (size_t)(lane_row - 1) * N +
                                             (ltid + (c / VP) * TC) * VW + 2 * (c % VP)) = acc[c];
        }
        named_barrier(1, THREADS);
        if (lane_row == 0) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                for (int l = 1; l < RL; ++l)
                    acc[c] = add2(acc[c], *reinterpret_cast<const uint64_t*>(
                                              scr + (size_t)(l - 1) * N + (ltid + (c / VP) * TC) * VW +
                                              2 * (c % VP)));
        }
    }
    if (lane_row == 0) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            float* ov = out + (ltid + v * TC) * VW;
            if constexpr (VW % 4 == 0) {
#pragma unroll
                for (int k = 0; k < VW / 4; ++k)
                    reinterpret_cast<ulonglong2*>(ov)[k] =
                        make_ulonglong2(acc[v * VP + 2 * k], acc[v * VP + 2 * k + 1]);
            } else {
                *reinterpret_cast<uint64_t*>(ov) = acc[v];
            }
        }
    }
    // ||r||^2: one double-single value per row lane (held by ltid == 0)
    if (ltid == 0) dred[lane_row] = r2;
    named_barrier(1, THREADS);
    if (tid == 0) {
        float2 s = dred[0];
        for (int l = 1; l < RL; ++l) s = ds_add(s, dred[l]);
        r2part[blockIdx.x] = s;
        // without the grid barrier below, the last block to arrive sums the partials
        sflag[0] = (g_out == nullptr && last_block_arrive(&ctrl->ticket_prod)) ? 1 : 0;
    }
    named_barrier(1, THREADS);
    // ||r||^2 = sum of the G partials with all warps (G <= THREADS), fixed order
    auto sum_r2 = [&]() {
        float2 v = tid < G ? __ldcg(r2part + tid) : make_float2(0.f, 0.f);
        v = warp_sum_ds(v);
        if ((tid & 31) == 0) dred[tid >> 5] = v;
        named_barrier(1, THREADS);
        if (tid == 0) {
            float2 t = dred[0];
            for (int w = 1; w < S::WARPS; ++w) t = ds_add(t, dred[w]);
            ctrl->r2 = ds_value(t);
        }
    };
    if (sflag[0]) sum_r2();
    if (g_out == nullptr) return;

    // ---------------- grid barrier, then g = sum of the G partials ----------------
    // All G blocks are co-resident (cooperative launch, one block per SM), so
    // a bounded spin on a monotone arrival counter is a grid barrier.
    named_barrier(1, THREADS);
    if (tid == 0) {
        __threadfence();
        const unsigned long long t = atomicAdd(&ctrl->gbar, 1ull);
        // bar_extra (0 outside the timeout test) raises the target beyond what the
        // grid's arrivals reach, so that only this bounded spin runs out
        const unsigned long long target =
            (t / (unsigned long long)G + 1ull) * (unsigned long long)G + (unsigned)bar_extra;
        const long long t0 = clock64();
        while (ld_acquire_u64(&ctrl->gbar) < target) {
            if (clock64() - t0 > budget) {
                set_error(ctrl, ERR_TIMEOUT, host_err);
                break;
            }
        }
        __threadfence();
    }
    named_barrier(1, THREADS);
    if (blockIdx.x == 0) sum_r2();   // every block's partial is visible after the barrier
    // This block's slice of float4 columns; warp w sums partials w, w+WARPS, ... and
    // warp 0 adds the warp sums in order (deterministic).
    const int N4 = N / 4;
    const int c0 = (int)(((long long)N4 * blockIdx.x) / G);
    const int c1 = (int)(((long long)N4 * (blockIdx.x + 1)) / G);
    const float4* gp4 = reinterpret_cast<const float4*>(gpart);
    float4* sred = reinterpret_cast<float4*>(smem);   // [WARPS][32], the stage ring is free
    float4* g4 = reinterpret_cast<float4*>(g_out);
    const int lane = tid & 31, warp = tid >> 5;
    constexpr int NWC = S::WARPS;
    constexpr int BATCH = (160 + NWC - 1) / NWC;   // partials in flight per thread (G <= 160: one round)
    for (int base = c0; base < c1; base += 32) {
        const int c = base + lane;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < c1) {
            for (int p0 = warp; p0 < G; p0 += NWC * BATCH) {
                float4 v[BATCH];
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {   // all loads issued before the first add
                    const int p = p0 + k * NWC;
                    v[k] = p < G ? __ldcg(gp4 + (size_t)p * N4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {   // partials in increasing order
                    s.x += v[k].x; s.y += v[k].y; s.z += v[k].z; s.w += v[k].w;
                }
            }
        }
        sred[warp * 32 + lane] = s;
        named_barrier(1, THREADS);
        if (warp == 0 && c < c1) {
            float4 t = sred[lane];
#pragma unroll
            for (int w = 1; w < NWC; ++w) {
                const float4 v = sred[w * 32 + lane];
                t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
            }
            g4[c] = t;
        }
        named_barrier(1, THREADS);
    }
}

// ---------------------------------------------------------------------------
// Shape table: (precision, n) -> (TC, VW, V, RL, RB, NST), and the rows a block
// takes at least.  N = n^2 = TC VW V.
// ---------------------------------------------------------------------------
template <int PREC, int TC, int VW, int V, int RL, int RB, int NST>
static cudaError_t launch_prod_t(int grid, const ProdArgs& a, cudaStream_t s)
{
    using S = ProdShape<PREC, TC, VW, V, RL, RB, NST>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(S::THREADS, 1, 1);
    cfg.dynamicSmemBytes = S::SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (a.g_out) {   // the grid barrier needs co-resident blocks
        attr[na].id = cudaLaunchAttributeCooperative;
        attr[na].val.cooperative = 1;
        ++na;
    }
    if (a.pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    const int pf = (int)(PROD_PF_BYTES / S::STAGE);
    auto kernel = (a.m + grid - 1) / grid > S::YMAX ? k_products<PREC, TC, VW, V, RL, RB, NST, true>
                                                    : k_products<PREC, TC, VW, V, RL, RB, NST, false>;
    return cudaLaunchKernelEx(&cfg, kernel, a.P0, a.P1, a.rscale, a.m, a.x, a.y, a.r, a.gpart, a.g_out,
                              a.r2part, a.ctrl, a.mode, (cudaGraphConditionalHandle)a.cond, a.set_cond,
                              a.budget, pf, a.bar_extra, a.host_err);
}

template <int PREC, int TC, int VW, int V, int RL, int RB, int NST>
static cudaError_t configure_t()
{
    using S = ProdShape<PREC, TC, VW, V, RL, RB, NST>;
    for (auto kernel : {k_products<PREC, TC, VW, V, RL, RB, NST, false>, k_products<PREC, TC, VW, V, RL, RB, NST, true>}) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// (n = 48, binary32: 8 rows a step in two row lanes; 4 rows on 384 x 6 columns were slower from
// m = 1152 on: 10.2, 14.3, 43.8 us a launch at m = 1152, 4700, 20000, here 9.8, 12.3, 36.8.)
//    precision, n, minimum rows per block, TC, VW, V, RL, RB, NST
#define TVCS_PROD_TABLE(X)                \
    X(0, 16, 8, 64, 4, 1, 8, 2, 4)        \
    X(0, 32, 4, 256, 4, 1, 2, 4, 4)       \
    X(0, 48, 4, 192, 4, 3, 2, 4, 3)       \
    X(0, 64, 2, 512, 4, 2, 1, 4, 3)       \
    X(0, 96, 1, 512, 2, 9, 1, 2, 3)       \
    X(0, 128, 1, 512, 4, 8, 1, 1, 3)      \
    X(1, 32, 4, 256, 4, 1, 2, 4, 4)       \
    X(1, 64, 2, 512, 8, 1, 1, 4, 3)       \
    X(1, 128, 1, 512, 8, 4, 1, 1, 3)      \
    X(2, 32, 4, 256, 4, 1, 2, 4, 4)       \
    X(2, 64, 2, 512, 8, 1, 1, 4, 4)       \
    X(2, 128, 1, 512, 8, 4, 1, 1, 4)

bool prod_supported(int prec, int n)
{
#define X(PR, NN, MR, TC, VW, V, RL, RB, NST) \
    if (prec == PR && n == NN) return true;
    TVCS_PROD_TABLE(X)
#undef X
    return false;
}

int prod_grid(int prec, int n, int m, int num_sms)
{
    int mr = 1;
#define X(PR, NN, MR, TC, VW, V, RL, RB, NST) \
    if (prec == PR && n == NN) mr = MR;
    TVCS_PROD_TABLE(X)
#undef X
    const int g = (m + mr - 1) / mr;
    const int cap = num_sms > 32 ? num_sms - 16 : num_sms;   // 16 SMs stay free for the u-solve cluster
    return g < cap ? g : cap;
}

cudaError_t prod_configure(int prec, int n)
{
#define X(PR, NN, MR, TC, VW, V, RL, RB, NST) \
    if (prec == PR && n == NN) return configure_t<PR, TC, VW, V, RL, RB, NST>();
    TVCS_PROD_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t launch_products(int prec, int n, int grid, const ProdArgs& a, cudaStream_t s)
{
#define X(PR, NN, MR, TC, VW, V, RL, RB, NST) \
    if (prec == PR && n == NN) return launch_prod_t<PR, TC, VW, V, RL, RB, NST>(grid, a, s);
    TVCS_PROD_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Gather of the partials, normalisation, fill.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_gather(const float* __restrict__ gpart, int P, int N,
                                                float scale, float* __restrict__ out,
                                                double* __restrict__ part, Ctrl* __restrict__ ctrl)
{
    __shared__ double red[32];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double sq = 0.0;
    if (i < N) {
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        int p = 0;
        for (; p + 4 <= P; p += 4) {
            s0 += gpart[(size_t)p * N + i];
            s1 += gpart[(size_t)(p + 1) * N + i];
            s2 += gpart[(size_t)(p + 2) * N + i];
            s3 += gpart[(size_t)(p + 3) * N + i];
        }
        for (; p < P; ++p) s0 += gpart[(size_t)p * N + i];
        const float v = scale * ((s0 + s1) + (s2 + s3));
        out[i] = v;
        sq = (double)v * (double)v;
    }
    const double s = block_sum(sq, red);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    __shared__ int is_last;
    if (!last_block_all(&ctrl->ticket_gather, &is_last)) return;
    const double t = block_sum_array(part, gridDim.x, 1, red);
    if (threadIdx.x == 0) ctrl->vec2 = t;
}

// g = sum over the P per-block partials, in a fixed order.  A block covers 32
// float4 columns with 8 partial slices (one warp each); slice k sums partials
// k, k+8, ..., then slice 0 adds the 8 slice sums in order.
__global__ void __launch_bounds__(256) k_greduce(const float4* __restrict__ gpart, int P, int N4,
                                                 float4* __restrict__ g,
                                                 const Ctrl* __restrict__ ctrl, int mode)
{
    __shared__ float4 acc[8][32];
    if (mode == MODE_ITER && ctrl->skip) return;
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < N4) {
        for (int p = slice; p < P; p += 8) {
            const float4 v = gpart[(size_t)p * N4 + c];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
    }
    acc[slice][lane] = s;
    __syncthreads();
    if (slice == 0 && c < N4) {
        float4 t = acc[0][lane];
#pragma unroll
        for (int k = 1; k < 8; ++k) {
            const float4 v = acc[k][lane];
            t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
        }
        g[c] = t;
    }
}

cudaError_t launch_greduce(const float* gpart, int P, int N, float* g, const Ctrl* ctrl, int mode,
                           cudaStream_t s)
{
    const int N4 = N / 4;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((N4 + 31) / 32, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, k_greduce, reinterpret_cast<const float4*>(gpart), P, N4,
                              reinterpret_cast<float4*>(g), ctrl, mode);
}

__global__ void k_normalize(const float* __restrict__ z, float* __restrict__ v, int N,
                            const Ctrl* __restrict__ ctrl)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double nrm = sqrt(ctrl->vec2);
    if (i < N) v[i] = (float)((double)z[i] / nrm);
}

__global__ void k_fill(float* __restrict__ v, int N, float value)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) v[i] = value;
}

// Start of a run: the loop bookkeeping of the control block, set on the device
// (no host round trip before the loop); the other fields keep their values.
__global__ void k_run_begin(Ctrl* __restrict__ c, int max_iter, int loops_max, double tol, int algo)
{
    c->it = 0;
    c->max_iter = max_iter;
    c->done = 0;
    c->skip = 0;
    c->stop_by_tol = 0;
    c->loops = 0;
    c->loops_max = loops_max;
    c->tol = tol;
    c->error = 0;
    c->algo = algo;
    c->lbar = 0ull;
    c->ticket_fft = c->ticket_prod = c->ticket_fin = c->ticket_w = c->ticket_gather = 0u;
}

// Start point of a solve, on the device (no host round trip).
__global__ void k_init_state(Ctrl* __restrict__ c, float* __restrict__ w, float* __restrict__ lam, int N,
                             int given)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (given) {   // w^0 = 0 in the current copy; u and lambda are the caller's
        const int par = c->wpar;
        if (i < 2 * N) w[(size_t)par * 2 * N + i] = 0.f;
    } else if (i < 4 * N) {
        w[i] = 0.f;
        lam[i] = 0.f;
    }
    if (i == 0) {
        c->pending = 0;
        if (!given) c->wpar = 0;
        c->error = 0;
    }
}

void launch_init_state(Ctrl* c, float* w, float* lam, int N, int given, cudaStream_t s)
{
    k_init_state<<<(4 * N + 255) / 256, 256, 0, s>>>(c, w, lam, N, given);
}

void launch_run_begin(Ctrl* c, int max_iter, int loops_max, double tol, int algo, cudaStream_t s)
{
    k_run_begin<<<1, 1, 0, s>>>(c, max_iter, loops_max, tol, algo);
}

void launch_gather(const float* gpart, int P, int N, float scale, float* out, double* part,
                   Ctrl* ctrl, cudaStream_t s)
{
    k_gather<<<(N + 255) / 256, 256, 0, s>>>(gpart, P, N, scale, out, part, ctrl);
}

void launch_normalize(const float* z, float* v, int N, const Ctrl* ctrl, cudaStream_t s)
{
    k_normalize<<<(N + 255) / 256, 256, 0, s>>>(z, v, N, ctrl);
}

void launch_fill(float* v, int N, float value, cudaStream_t s)
{
    k_fill<<<(N + 255) / 256, 256, 0, s>>>(v, N, value);
}

}  // namespace tvcs
