// The whole iteration loop of one problem (Algorithm 2 or 1; rows a1-a7 of every
// iteration and the test of eq. (stop)) as ONE persistent cooperative launch, for images
// up to 96 x 96 with a stored A (Xiao & Yang, Sec. 2.1-2.2).
//
// G blocks, one per SM.  Block b owns a contiguous range of rows of A for the two products.  At
// n <= 64 these stay on chip for the whole launch where they fit, as binary32: 8 to 32 of them in
// registers, the rest in shared memory (k_loop_reg).  Otherwise (k_loop) they come through a
// ring of pieces filled by bulk copies, as in k_products.cu.  The first n/2 blocks also carry the u-step: block j owns the
// image rows 2j and 2j+1 and column slot j of the half spectrum (slot 0: the two real
// columns 0 and n/2 packed as one complex column).  An iteration:
//   1  blocks j: lambda update, shrink and D^T y of their rows (one halo row recomputed),
//      g of their rows as the sum of the G blocks' partials of A^T r, right-hand side,
//      one packed row transform (one warp), half spectra sent to the column slots' blocks;
//   2  blocks j: column transform, divide, inverse, rows sent back; inverse row
//      transform, u <- u + d sent to every block, norms of eq. (stop);
//   3  all blocks: u into registers, the products over their rows, partial of A^T r to
//      global memory, arrival on a counter that the blocks j wait for (step 1);
//   4  all blocks: eq. (stop) from the n/2 blocks' norms, the same sums in the same order
//      everywhere, so that every block leaves in the same iteration.
// Values sent between blocks travel as 8-byte words of a binary32 value and a tag (the
// iteration's number): the reader polls the words themselves, so an exchange costs one
// store and one load through L2 and no fence or flag.  The buffers alternate between
// iterations; a buffer is written again only after its readers have passed a later exchange.
//
// What bounds it: the exchanges between blocks (1 to 1.5 us each through L2: partials, column
// slots, rows, u), and at n = 96 reading A.  The chain of two launches per iteration that it
// replaces (u-solve cluster, products) paid two kernel boundaries, a grid barrier with a
// global reduction and a second read of g, and had loop graphs to build.  us an iteration, 200
// iterations, binary32, as the chain -> k_loop -> k_loop_reg:
//   n = 16 (m = 77) 9.6 -> 6.7 -> 4.8, n = 32 (307) 11.7 -> 7.8 -> 7.3, n = 48 (691) 12.5 -> 8.7 ->
//   8.0, n = 64 (1229) 14.75 -> 11.4 -> 9.7 (2048: 13.2 -> 10.0; fp8, 1229: 13.8 -> 9.7), n = 96
//   (921) 17.0 -> 16.3, n = 96 (2765) 23.7 -> 23.3.
// (k_loop_reg varies by where the exchange buffers lie on the two dies: over devices and handles
// n = 16 4.8-6.1, n = 32 6.0-9.3, n = 48 8.0-9.0, n = 64 9.2-12.5.)
// (From the ring a pass over 9 rows took three steps of 1.3 us, each a wait, a decode, a warp
// reduction and a block barrier in series; from registers all rows share one of each.)  At
// n = 128 k_loop measured 52.5 us against 52.1 (u-solve and exchanges take 13 us in which L2 cannot
// hold more of A than the row order already keeps there), so that size keeps the chain.
//
// What it costs others: the launch holds its SMs (all of them at n = 96 and at n = 64 from m = 1209
// on) for the whole run, where the chain gave them back every iteration.  Two threads with a
// handle each, ms a call: 64 x 64 (m = 1229), 300 iterations, alone 3.3 (chain 4.6), both at once
// 6.5 (6.1); 64 x 64, 20 iterations, next to runs of 300 at 96 x 96 5.1 (0.73).
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "kernels.h"
#include "loop_exchange.cuh"
#include "loop_rows.cuh"
#include "products.cuh"
#include "usolve_steps.cuh"

namespace tvcs {

namespace {

// A block's scalars, in shared memory: what a section needs it reads again, so that no value
// stays in a register through the products' loop (at n = 128 its rows, u and sums take 96 of
// the 128; kept values spilled 25 registers into that loop, which made it twice as slow).
struct LoopState {
    int gave_up;             // a wait ran out
    int end;                 // 0, or why the run ends: 1 iterations, 2 eq. (stop), 3 not finite
    int pending;             // the multiplier update of the last u is due
    int algo;
    int i0, nrows;           // this block's rows of A
    int last;                // this block is the last to end
    double du2, u2, tol;     // norms of the last iteration, eq. (stop)
};

// The ring of A in shared memory, in pieces of RP rows.  Thread 0 issues the pieces of pass
// after pass (a pass reads every row of the block once), odd passes from the last piece to
// the first: the rows read last are then the next pass's first, and partly still in L2
// (n = 96, m = 2765: 24.2 -> 23.3 us an iteration).  A block whose rows fit in the ring copies
// them once.
struct Ring {
    const unsigned char *p0, *p1;   // the block's rows in the planes of A
    uint64_t pol;
    int nrows, pieces, passes;        // passes to issue (1 where the ring holds every row)
    int pass, o, slot, phase;         // next piece to issue, its slot and the slot's phase
};

template <int NN_, int PREC_, int TC_, int VW_, int V_, int RL_, int RB_, int RP_, int NPC_>
struct LoopShape {
    using P = ProdShape<PREC_, TC_, VW_, V_, RL_, RB_, 2>;
    static_assert(P::N == NN_ * NN_, "columns");
    static constexpr int NN = NN_, PREC = PREC_, TC = TC_, VW = VW_, V = V_, RL = RL_, RB = RB_, RREG = 0;
    static constexpr int CP = P::CPT / 2;
    static constexpr int N = P::N, THREADS = P::THREADS, WARPS = P::WARPS, RS = P::RS, WPR = P::WPR;
    static constexpr int B0 = P::B0, B1 = P::B1;
    static constexpr int RP = RP_, Q = RS / RP, NPC = NPC_;   // rows a piece, pieces a step, pieces in the ring
    static_assert(RS % RP == 0 && (Q == 1 || (RL == 1 && RP == 1)), "a step's rows in its pieces");
    static constexpr size_t P1_OFF = (size_t)RP * N * B0, PIECE = (size_t)RP * N * (B0 + B1);
    static constexpr int NP = NN / 2;             // row pairs = column slots = blocks of the u-step
    static constexpr int GC = 2 * NN / 4;         // float4 columns of a row pair
    static constexpr int GG = THREADS / GC;       // groups of partials in the sum of g
    static constexpr int YMAX = 512;              // rows of y (and scales) kept in shared memory
    static constexpr int WL = 3 * NN;             // rows 2j-1, 2j, 2j+1
    static constexpr size_t al(size_t b) { return (b + 15) / 16 * 16; }
    static constexpr size_t O_BAR = NPC * PIECE;
    static constexpr size_t O_RED = O_BAR + al(NPC * 8);
    static constexpr size_t O_DRED = O_RED + al(2 * RS * WPR * 4);         // [32] float2
    static constexpr size_t O_STATE = O_DRED + 32 * 8;
    static constexpr size_t O_RING = O_STATE + al(sizeof(LoopState));
    static constexpr size_t O_Y = O_RING + al(sizeof(Ring));
    static constexpr size_t O_S = O_Y + YMAX * 4;
    static constexpr size_t O_SU = O_S + (PREC == 2 ? YMAX * 4 : 0);      // u rows 2j-1 .. 2j+2
    static constexpr size_t O_WL = O_SU + 4 * NN * 4;                      // 2 x (w1, w2, l1, l2) x 3 rows
    static constexpr size_t O_Y1 = O_WL + 2 * 4 * WL * 4;                  // rows 2j, 2j+1
    static constexpr size_t O_Y2 = O_Y1 + 2 * NN * 4;                      // rows 2j-1 .. 2j+1
    static constexpr size_t O_G = O_Y2 + 3 * NN * 4;                       // g of rows 2j, 2j+1
    static constexpr size_t O_GS = O_G + 2 * NN * 4;                       // [GG][GC] float4
    static constexpr size_t GS = (size_t)GG * GC * 16;
    static constexpr size_t O_FA = O_GS + GS;                              // two transforms
    static constexpr size_t O_FB = O_FA + NN * 8;
    static constexpr size_t O_TW = O_FB + NN * 8;
    static constexpr size_t O_RD = O_TW + NN * 8;                          // rdiv of the slot and of column n/2
    static constexpr size_t SMEM = O_RD + 2 * NN * 4;
    static_assert(GG >= 1 && THREADS % 32 == 0 && THREADS >= 96 && NN % 4 == 0, "threads");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// The same without a ring: every row of A on chip as binary32 for the whole launch, RL RREG of
// them in registers (a thread has its columns of RREG rows), up to XMAX more in shared memory.
template <int NN_, int TC_, int V_, int RL_, int RREG_>
struct RegShape {
    static constexpr int NN = NN_, PREC = 0, TC = TC_, VW = 4, V = V_, RL = RL_, RREG = RREG_;
    static constexpr int N = NN * NN, THREADS = TC * RL, WARPS = THREADS / 32, WPR = TC / 32, CP = VW * V / 2;
    static_assert(TC * VW * V == N && TC % 32 == 0 && RREG % 4 == 0 && THREADS >= 96 && THREADS <= 512, "split");
    static constexpr int NP = NN / 2, GC = 2 * NN / 4, GG = THREADS / GC, WL = 3 * NN;
    static constexpr int RROWS = RL * RREG;
    static constexpr int RED = WPR | 1;           // stride of a row's warp sums (odd banks)
    static constexpr size_t al(size_t b) { return (b + 15) / 16 * 16; }
    static constexpr size_t O_DRED = 0;           // [32] float2
    static constexpr size_t O_STATE = O_DRED + 32 * 8;
    static constexpr size_t O_SU = O_STATE + al(sizeof(LoopState));       // as in LoopShape
    static constexpr size_t O_WL = O_SU + 4 * NN * 4;
    static constexpr size_t O_Y1 = O_WL + 2 * 4 * WL * 4;
    static constexpr size_t O_Y2 = O_Y1 + 2 * NN * 4;
    static constexpr size_t O_G = O_Y2 + 3 * NN * 4;
    static constexpr size_t O_GS = O_G + 2 * NN * 4;
    static constexpr size_t GS = std::max((size_t)GG * GC * 16, (size_t)(RL - 1) * N * 4);
    static constexpr size_t O_FA = O_GS + GS;
    static constexpr size_t O_FB = O_FA + NN * 8;
    static constexpr size_t O_TW = O_FB + NN * 8;
    static constexpr size_t O_RD = O_TW + NN * 8;
    static constexpr size_t O_RED = O_RD + 2 * NN * 4;
    static constexpr size_t ROW_BYTES = (size_t)RED * 4 + 8;   // a row's warp sums, r and f
    static constexpr size_t LIMIT = 227 * 1024;
    static constexpr int XMAX = (int)((LIMIT - O_RED - 64 - RROWS * ROW_BYTES) / ((size_t)N * 4 + ROW_BYTES));
    static constexpr int RMAX = RROWS + XMAX, YMAX = RMAX;
    static constexpr size_t O_R = al(O_RED + (size_t)RMAX * RED * 4);
    static constexpr size_t O_Y = al(O_R + (size_t)RMAX * 4);
    static constexpr size_t O_A = al(O_Y + (size_t)RMAX * 4);
    static constexpr size_t smem(int rows) { return O_A + (size_t)std::max(0, rows - RROWS) * N * 4; }
    static_assert(GG >= 1 && smem(RMAX) <= LIMIT, "shared memory");
};

#define LOOP_SMEM extern __shared__ __align__(128) unsigned char smem[]
#define LOOP_AT(T, off) reinterpret_cast<T*>(smem + (off))

// One thread: until the counter reaches `target`; what was written before the arrivals is
// then visible.
__device__ __forceinline__ void loop_wait_count(const unsigned long long* c, unsigned long long target,
                                                const Waits& w)
{
    const long long t0 = clock64();
    while (ld_acquire_u64(c) < target) {
        if (*w.gave_up) break;
        if (clock64() - t0 > w.budget) {
            *w.gave_up = 1;
            break;
        }
    }
    __threadfence();
}

template <class S>
__device__ __forceinline__ void ring_issue()   // thread 0; nothing past the last pass
{
    LOOP_SMEM;
    Ring& g = *LOOP_AT(Ring, S::O_RING);
    uint64_t* full = LOOP_AT(uint64_t, S::O_BAR);
    const int pass = g.pass, o = g.o, slot = g.slot;
    if (pass >= g.passes) return;
    const int b0 = ((pass & 1) ? g.pieces - 1 - o : o) * S::RP;
    const uint32_t ent = (uint32_t)min(S::RP, g.nrows - b0) * S::N;
    unsigned char* dst = smem + (size_t)slot * S::PIECE;
    mbar_arrive_expect_tx(&full[slot], ent * (S::B0 + S::B1));
    tma_load_1d(dst, g.p0 + (size_t)b0 * S::N * S::B0, ent * S::B0, &full[slot], g.pol);
    if constexpr (S::B1 > 0)
        tma_load_1d(dst + S::P1_OFF, g.p1 + (size_t)b0 * S::N * S::B1, ent * S::B1, &full[slot], g.pol);
    const bool last = o + 1 == g.pieces, wrap = slot + 1 == S::NPC;
    g.pass = last ? pass + 1 : pass;
    g.o = last ? 0 : o + 1;
    g.slot = wrap ? 0 : slot + 1;
    if (wrap) g.phase ^= 1;
}

// a1-a3 up to y = beta (w - D u) - lambda of the rows 2j-1 (y2 only), 2j, 2j+1, by the
// `cnt` threads from t = 0; w and lambda go from copy `from` to the other one.
template <class S>
__device__ __forceinline__ void loop_shrink(float beta, int from, int t, int cnt)
{
    LOOP_SMEM;
    constexpr int NN = S::NN, WL = S::WL;
    const float* su = LOOP_AT(float, S::O_SU);
    float* sy1 = LOOP_AT(float, S::O_Y1);
    float* sy2 = LOOP_AT(float, S::O_Y2);
    const float* src = LOOP_AT(float, S::O_WL) + from * 4 * WL;
    float* dst = LOOP_AT(float, S::O_WL) + (from ^ 1) * 4 * WL;
    const float inv_beta = 1.0f / beta;
    const int pending = LOOP_AT(LoopState, S::O_STATE)->pending;
    for (int i = t; i < WL; i += cnt) {
        const int rr = i / NN, c = i - rr * NN;
        const int cp = (c + 1 == NN) ? 0 : c + 1;
        const float uc = su[i];
        const float d1 = su[rr * NN + cp] - uc, d2 = su[i + NN] - uc;
        float l1 = src[2 * WL + i], l2 = src[3 * WL + i];
        if (pending) {   // eq. (udlamb) for the previous iteration
            l1 -= beta * (src[i] - d1);
            l2 -= beta * (src[WL + i] - d2);
        }
        const float z1 = d1 + l1 * inv_beta, z2 = d2 + l2 * inv_beta;
        const float nz = sqrtf(z1 * z1 + z2 * z2);
        float w1 = 0.0f, w2 = 0.0f;
        if (nz > inv_beta) {
            const float s = (nz - inv_beta) / nz;
            w1 = s * z1;
            w2 = s * z2;
        }
        sy2[i] = beta * (w2 - d2) - l2;
        if (rr >= 1) sy1[i - NN] = beta * (w1 - d1) - l1;
        dst[i] = w1;
        dst[WL + i] = w2;
        dst[2 * WL + i] = l1;
        dst[3 * WL + i] = l2;
    }
}

// The u-step of block j (one warp): right-hand side, row transform, column slot j, inverse
// row transform, the new u of rows 2j, 2j+1 to every block, norms.
template <class S>
__device__ __forceinline__ void loop_ustep(const LoopArgs& q, int it)
{
    LOOP_SMEM;
    constexpr int NN = S::NN, NP = S::NP, N = S::N;
    const int lane = fresh_tid() & 31;
    const int blk = blockIdx.x, r0 = 2 * blk, half = it & 1;
    const uint32_t tag = q.tag0 + (uint32_t)it;
    LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    const Waits waits{q.budget, &st->gave_up};
    const float* su = LOOP_AT(float, S::O_SU);
    const float* sy1 = LOOP_AT(float, S::O_Y1);
    const float* sy2 = LOOP_AT(float, S::O_Y2);
    const float* sg = LOOP_AT(float, S::O_G);
    float2* fa = LOOP_AT(float2, S::O_FA);
    float2* fb = LOOP_AT(float2, S::O_FB);
    const float2* tw = LOOP_AT(float2, S::O_TW);
    const float* rdiv = LOOP_AT(float, S::O_RD);
    uint64_t* colx = q.colx + (size_t)half * NP * NN * 2;
    uint64_t* rowx = q.rowx + (size_t)half * NN * NP * 2;
    uint64_t* ubuf = q.ubuf + (size_t)half * N;
    if (lane == 0) st->pending = st->algo == 0 ? 1 : 0;   // u is about to move
    // a3: right-hand side of the two rows as one complex sequence
    for (int c = lane; c < NN; c += 32) {
        const int cm = (c == 0) ? NN - 1 : c - 1;
        float v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float dty = sy1[h * NN + cm] - sy1[h * NN + c] + sy2[h * NN + c] - sy2[(h + 1) * NN + c];
            v[h] = dty - q.mu * sg[h * NN + c];
        }
        fa[c] = make_float2(v[0], v[1]);
    }
    __syncwarp();
    const float2* Z = fft_warp<NN, false>(fa, fb, tw, lane);
    // half spectra of the two rows to the column slots' blocks
    for (int s = lane; s < NP; s += 32) {
        const float2 a = Z[s], b = Z[(NN - s) % NN];
        uint64_t* dst = colx + ((size_t)s * NN + r0) * 2;
        if (s == 0) {
            const float2 n2 = Z[NN / 2];
            send2(dst, a.x, n2.x, tag);
            send2(dst + 2, a.y, n2.y, tag);
        } else {
            send2(dst, 0.5f * (a.x + b.x), 0.5f * (a.y - b.y), tag);
            send2(dst + 2, 0.5f * (a.y + b.y), -0.5f * (a.x - b.x), tag);
        }
    }
    __syncwarp();
    // a4: column slot j
    {
        constexpr int K = (NN + 31) / 32;
        ulonglong2 v[K];
        const uint64_t* src = colx + (size_t)blk * NN * 2;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k < NN) v[k] = peek2(src + 2 * (lane + 32 * k));
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (lane + 32 * k < NN) {
                v[k] = await2(src + 2 * (lane + 32 * k), tag, v[k], waits);
                fa[lane + 32 * k] = make_float2(word_f(v[k].x), word_f(v[k].y));
            }
    }
    __syncwarp();
    float2* X = fft_warp<NN, false>(fa, fb, tw, lane);
    if (blk != 0) {
        for (int p = lane; p < NN; p += 32) {
            const float rd = rdiv[p];
            X[p] = make_float2(X[p].x * rd, X[p].y * rd);
        }
    } else {   // columns 0 and n/2, separated by conjugate symmetry
        for (int k = lane; 2 * k <= NN; k += 32) {
            const int km = (NN - k) % NN;
            const float2 zk = X[k], zm = X[km];
            const float a0 = rdiv[k], an = rdiv[NN + k];
            const float2 c0 = make_float2(0.5f * (zk.x + zm.x) * a0, 0.5f * (zk.y - zm.y) * a0);
            const float2 cn = make_float2(0.5f * (zk.y + zm.y) * an, -0.5f * (zk.x - zm.x) * an);
            X[k] = make_float2(c0.x - cn.y, c0.y + cn.x);
            if (km != k) X[km] = make_float2(c0.x + cn.y, cn.x - c0.y);
        }
    }
    __syncwarp();
    const float2* Y = fft_warp<NN, true>(X, X == fa ? fb : fa, tw, lane);
    for (int p = lane; p < NN; p += 32) send2(rowx + ((size_t)p * NP + blk) * 2, Y[p].x, Y[p].y, tag);
    __syncwarp();
    // the rows' half spectra, packed for one inverse transform
    {
        constexpr int K = (NP + 31) / 32;
        ulonglong2 v[2][K];
        const uint64_t* src = rowx + (size_t)r0 * NP * 2;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (lane + 32 * k < NP) v[h][k] = peek2(src + 2 * (h * NP + lane + 32 * k));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int s = lane + 32 * k;
            if (s >= NP) continue;
            const ulonglong2 vx = await2(src + 2 * s, tag, v[0][k], waits);
            const ulonglong2 vy = await2(src + 2 * (NP + s), tag, v[1][k], waits);
            const float2 Xv = make_float2(word_f(vx.x), word_f(vx.y));
            const float2 Yv = make_float2(word_f(vy.x), word_f(vy.y));
            if (s == 0) {
                fa[0] = make_float2(Xv.x, Yv.x);
                fa[NN / 2] = make_float2(Xv.y, Yv.y);
            } else {
                fa[s] = make_float2(Xv.x - Yv.y, Xv.y + Yv.x);
                fa[NN - s] = make_float2(Xv.x + Yv.y, Yv.x - Xv.y);
            }
        }
    }
    __syncwarp();
    const float2* z = fft_warp<NN, true>(fa, fb, tw, lane);
    // u <- u + d, sent to every block; then the norms of eq. (stop)
    const float sc = 1.0f / (float)(NN * NN);
    for (int c = 2 * lane; c < NN; c += 64) {
        const float2 za = z[c], zb = z[c + 1];
        send2(ubuf + r0 * NN + c, su[NN + c] + za.x * sc, su[NN + c + 1] + zb.x * sc, tag);
        send2(ubuf + (r0 + 1) * NN + c, su[2 * NN + c] + za.y * sc, su[2 * NN + c + 1] + zb.y * sc, tag);
    }
    float2 du2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
    for (int c = lane; c < NN; c += 32) {
        const float2 v = z[c];
        du2 = ds_add(du2, ds_sq(v.x * sc));
        u2 = ds_add(u2, ds_sq(su[NN + c]));
        du2 = ds_add(du2, ds_sq(v.y * sc));
        u2 = ds_add(u2, ds_sq(su[2 * NN + c]));
    }
    du2 = warp_sum_ds(du2);
    u2 = warp_sum_ds(u2);
    if (lane == 0) {
        uint64_t* nb = q.nbuf + ((size_t)half * NP + blk) * 4;
        send2(nb, du2.x, du2.y, tag);
        send2(nb + 2, u2.x, u2.y, tag);
    }
}

// u of iteration `it` into the thread's registers, and in the u-step's blocks the rows
// 2j-1 .. 2j+2 for the next w-step.
template <class S>
__device__ __forceinline__ void loop_take_u(const LoopArgs& q, int it, uint64_t* xu)
{
    LOOP_SMEM;
    constexpr int NN = S::NN, TC = S::TC, VW = S::VW, V = S::V, N = S::N;
    LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    const Waits waits{q.budget, &st->gave_up};
    const int tid = fresh_tid();
    const int ltid = tid % TC;
    const uint32_t tag = q.tag0 + (uint32_t)it;
    const uint64_t* ubuf = q.ubuf + (size_t)(it & 1) * N;
    {
        constexpr int W2 = VW / 2;   // two-word packets per vector
        const uint64_t* xb = ubuf + (size_t)ltid * VW;
        // one packet first: while u is awaited only that one is polled
        const ulonglong2 v0 = await2(xb, tag, peek2(xb), waits);
        xu[0] = pack2(word_f(v0.x), word_f(v0.y));
        constexpr int NV = V * W2;
        constexpr int BATCH = 8;
    #pragma unroll
        for (int b = 1; b < NV; b += BATCH) {
            ulonglong2 v[BATCH];
            auto look = [&]() {   // the batch's packets; true once every one has arrived
                bool all = true;
    #pragma unroll
                for (int k = 0; k < BATCH; ++k)
                    if (b + k < NV) v[k] = peek2(xb + (size_t)((b + k) / W2) * TC * VW + 2 * ((b + k) % W2));
    #pragma unroll
                for (int k = 0; k < BATCH; ++k)
                    if (b + k < NV) all = all && has_tag(v[k], tag);
                return all;
            };
            if (!look()) {
                const long long t0 = clock64();
                while (!look()) {
                    if (*waits.gave_up) break;
                    if (clock64() - t0 > waits.budget) {
                        *waits.gave_up = 1;
                        break;
                    }
                }
            }
    #pragma unroll
            for (int k = 0; k < BATCH; ++k)
                if (b + k < NV) xu[b + k] = pack2(word_f(v[k].x), word_f(v[k].y));
        }
    }
    if (blockIdx.x < S::NP) {   // rows 2j-1 .. 2j+2 for the next w-step (warp 0 has read the old ones)
        float* su = LOOP_AT(float, S::O_SU);
        const int r0 = 2 * blockIdx.x;
        __syncthreads();
        for (int i = 2 * tid; i < 4 * NN; i += 2 * S::THREADS) {
            const int rr = i / NN, c = i - rr * NN;
            const uint64_t* p = ubuf + ((r0 - 1 + rr + NN) % NN) * NN + c;
            const ulonglong2 v = await2(p, tag, peek2(p), waits);
            su[i] = word_f(v.x);
            su[i + 1] = word_f(v.y);
        }
    }
}

// The block's partial of A^T r to global memory.
template <class S>
__device__ __forceinline__ void loop_partial(const LoopArgs& q, uint64_t* acc)
{
    LOOP_SMEM;
    constexpr int TC = S::TC, VW = S::VW, V = S::V, RL = S::RL, N = S::N, VP = VW / 2;
    [[maybe_unused]] constexpr int CP = S::CP;
    const int tid = fresh_tid();
    const int lane_row = tid / TC;
    const int ltid = tid - lane_row * TC;
    if constexpr (RL > 1) {   // the row lanes' sums meet in the scratch of g
        float* scr = LOOP_AT(float, S::O_GS);
        static_assert((size_t)(RL - 1) * N * 4 <= S::GS, "the lanes' sums fit");
        if (lane_row > 0) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                *reinterpret_cast<uint64_t*>(scr + (size_t)(lane_row - 1) * N + (ltid + (c / VP) * TC) * VW +
                                             2 * (c % VP)) = acc[c];
        }
        __syncthreads();
        if (lane_row == 0) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                for (int l = 1; l < RL; ++l)
                    acc[c] = add2(acc[c],
                                  *reinterpret_cast<const uint64_t*>(scr + (size_t)(l - 1) * N +
                                                                     (ltid + (c / VP) * TC) * VW + 2 * (c % VP)));
        }
    }
    if (lane_row == 0) {
        float* out = q.gpart + (size_t)blockIdx.x * N;
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
}

// One pass: u into registers, r = A u - f and the partial of A^T r over this block's rows,
// to global memory.
template <class S>
__device__ __forceinline__ void loop_pass(const LoopArgs& q, int it)
{
    LOOP_SMEM;
    constexpr int PREC = S::PREC, TC = S::TC, VW = S::VW, V = S::V, RB = S::RB;
    constexpr int N = S::N, RS = S::RS, WPR = S::WPR, CP = S::P::CPT / 2, VP = VW / 2, Q = S::Q;
    uint64_t* full = LOOP_AT(uint64_t, S::O_BAR);
    float* red = LOOP_AT(float, S::O_RED);
    volatile LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    const Waits waits{q.budget, &st->gave_up};
    const int tid = fresh_tid();
    const int lane_row = tid / TC;
    const int ltid = tid - lane_row * TC;

    uint64_t xu[CP], acc[CP];
    loop_take_u<S>(q, it, xu);
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0ull;
    float2 r2 = make_float2(0.f, 0.f);   // double-single ||r||^2 of this lane's rows (ltid == 0)

    // ---------------- a6-a7 ----------------
    {
        const int nrows = st->nrows;
        const float* sy = LOOP_AT(float, S::O_Y);
        const float* ss = LOOP_AT(float, S::O_S);
        const int pieces = (nrows + S::RP - 1) / S::RP;
        const bool resident = pieces <= S::NPC, in_smem = nrows <= S::YMAX;
        const bool down = !resident && ((it - 1) & 1);   // from the last piece to the first
        // first piece to consume (a resident block's only phase has completed)
        const long long before = resident ? 0 : (long long)(it - 1) * pieces;
        int c_slot = (int)(before % S::NPC);
        uint32_t c_phase = (uint32_t)((before / S::NPC) & 1);
        // row b of this lane's step: li0 + b (pieces of a whole step), li0 +- b (pieces of one row)
        const int dli = down ? -RS : RS;
        int li0 = Q == 1 ? (down ? pieces - 1 : 0) * RS + lane_row * RB : (down ? nrows - 1 : 0);
        int left = nrows;   // rows of the pass still to come (Q > 1)
        for (int s = (nrows + RS - 1) / RS; s > 0; --s, li0 += dli, left -= RS) {
            int slot[Q];
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                slot[k] = c_slot;
                if (Q == 1 || k < left) {
                    const uint32_t ph = resident ? 0u : c_phase;
                    if (!mbar_try_wait(&full[c_slot], ph) && !*waits.gave_up &&
                        !mbar_wait(&full[c_slot], ph, q.budget))
                        *waits.gave_up = 1;
                    if (++c_slot == S::NPC) {
                        c_slot = 0;
                        c_phase ^= 1u;
                    }
                }
            }
            auto row_of = [&](int b) { return Q == 1 || !down ? li0 + b : li0 - b; };
            auto has_row = [&](int b) { return RS == 1 || (Q == 1 ? li0 + b < nrows : b < left); };
            uint64_t a[RB][CP];
            float* rb = red + ((s & 1) * RS + lane_row * RB) * WPR;
            float d[RB];
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                if (has_row(b)) {
                    const unsigned char* sb = smem + (size_t)slot[Q == 1 ? 0 : b] * S::PIECE;
                    const size_t row = Q == 1 ? (size_t)(lane_row * RB + b) * N : 0;
                    float sc = 1.f;
                    if constexpr (PREC == 2) sc = in_smem ? ss[row_of(b)] : q.rscale[st->i0 + row_of(b)];
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
                for (int b = 0; b < RB; ++b) rb[b * WPR + (ltid >> 5)] = d[b];
            }
            __syncthreads();   // the warps' parts are there, and nobody reads the pieces any more
            if (tid == 0 && !resident && !*waits.gave_up) {
#pragma unroll
                for (int k = 0; k < Q; ++k)   // as many as this step freed
                    if (Q == 1 || k < left) ring_issue<S>();
            }
#pragma unroll
            for (int b = 0; b < RB; ++b) {
                if (!has_row(b)) break;
                float dot;
                if constexpr (WPR % 4 == 0) {   // fixed tree over the warps' parts
                    uint64_t p[WPR / 4];
#pragma unroll
                    for (int w = 0; w < WPR / 4; ++w) {
                        const ulonglong2 t = reinterpret_cast<const ulonglong2*>(rb + b * WPR)[w];
                        p[w] = add2(t.x, t.y);
                    }
#pragma unroll
                    for (int o = 1; o < WPR / 4; o *= 2)
#pragma unroll
                        for (int w = 0; w + o < WPR / 4; w += 2 * o) p[w] = add2(p[w], p[w + o]);
                    const float2 t = unpack2(p[0]);
                    dot = t.x + t.y;
                } else {
                    dot = rb[b * WPR];
#pragma unroll
                    for (int w = 1; w < WPR; ++w) dot += rb[b * WPR + w];
                }
                const int li = row_of(b);
                const float ri = dot - (in_smem ? sy[li] : q.y[st->i0 + li]);
                if (ltid == 0) {
                    q.r[st->i0 + li] = ri;
                    r2 = ds_add(r2, ds_sq(ri));
                }
                const uint64_t rr = pack2(ri, ri);
#pragma unroll
                for (int c = 0; c < CP; ++c) acc[c] = fma2(rr, a[b][c], acc[c]);
            }
        }
    }

    if (ltid == 0) LOOP_AT(float2, S::O_DRED)[lane_row] = r2;
    loop_partial<S>(q, acc);
}

// The same pass over rows that stay on chip (RegShape).
template <class S>
__device__ __forceinline__ void loop_pass_reg(const LoopArgs& q, int it, const uint64_t (&a)[S::RREG][S::CP])
{
    LOOP_SMEM;
    const int nrows = *(volatile const int*)&LOOP_AT(LoopState, S::O_STATE)->nrows;
    const float* srow = LOOP_AT(float, S::O_A);
    float* sr = LOOP_AT(float, S::O_R);
    const int tid = fresh_tid(), lane_row = tid / S::TC, ltid = tid - lane_row * S::TC;
    uint64_t xu[S::CP], acc[S::CP];
    loop_take_u<S>(q, it, xu);
    reg_residual<S>(a, xu, srow, LOOP_AT(float, S::O_Y), LOOP_AT(float, S::O_RED), sr, nrows, tid);
    reg_adjoint<S>(a, srow, sr, nrows, lane_row, ltid, acc);
    loop_partial<S>(q, acc);
}

// After a pass: thread 0 arrives and, in the u-step's blocks, waits for all partials; warp 1
// decides eq. (stop); the other warps run the next w-step meanwhile (w and lambda of the
// other copy, in force only if the run goes on).
template <class S>
__device__ __forceinline__ void loop_arrive(const LoopArgs& q, int it)
{
    LOOP_SMEM;
    const int tid = fresh_tid(), lane = tid & 31, warp = tid >> 5;
    const int blk = blockIdx.x;
    const bool ublk = blk < S::NP;
    LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    const Waits waits{q.budget, &st->gave_up};
    if (warp == 0) {
        if (lane == 0) {
            if constexpr (S::RREG == 0) {
                const float2* dred = LOOP_AT(float2, S::O_DRED);
                float2 s = dred[0];
                for (int l = 1; l < S::RL; ++l) s = ds_add(s, dred[l]);
                q.r2part[blk] = s;
            }
            __threadfence();
            atomicAdd(&q.ctrl->lbar, 1ull);
            if (ublk) {
                loop_wait_count(&q.ctrl->lbar,
                                (unsigned long long)gridDim.x * (unsigned)it + (unsigned)q.bar_extra, waits);
            }
        }
    } else if (warp == 1) {
        float2 du2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
        for (int j = lane; j < S::NP; j += 32) {
            const uint64_t* nb = q.nbuf + ((size_t)(it & 1) * S::NP + j) * 4;
            const uint32_t tag = q.tag0 + (uint32_t)it;
            ulonglong2 a = peek2(nb), b = peek2(nb + 2);
            a = await2(nb, tag, a, waits);
            b = await2(nb + 2, tag, b, waits);
            du2 = ds_add(du2, make_float2(word_f(a.x), word_f(a.y)));
            u2 = ds_add(u2, make_float2(word_f(b.x), word_f(b.y)));
        }
        du2 = warp_sum_ds(du2);
        u2 = warp_sum_ds(u2);
        if (lane == 0) {
            const double tdu = ds_value(du2), tu = ds_value(u2), tol = st->tol;
            st->du2 = tdu;
            st->u2 = tu;
            int end = it >= q.iters ? 1 : 0;
            if (!isfinite(tdu) || !isfinite(tu))
                end = 3;
            else if (tol > 0.0 && (tu > 0.0 ? tdu <= tol * tol * tu : tdu == 0.0))
                end = 2;   // eq. (stop), reading C5
            st->end = end;
        }
    } else {
        if (ublk) loop_shrink<S>(q.beta, it & 1, tid - 64, S::THREADS - 64);
    }
}

// g of rows 2j, 2j+1: the G partials in GG groups, then the groups, fixed order.
template <class S>
__device__ __forceinline__ void loop_gather(const LoopArgs& q)
{
    LOOP_SMEM;
    constexpr int GC = S::GC, GG = S::GG;
    const int tid = fresh_tid(), G = gridDim.x;
    float4* sgs = LOOP_AT(float4, S::O_GS);
    const int col = tid % GC, grp = tid / GC;
    if (grp < GG) {
        const float4* gp = reinterpret_cast<const float4*>(q.gpart) + (size_t)2 * blockIdx.x * S::NN / 4 + col;
        constexpr int BATCH = S::RREG > 0 ? 152 / GG + 1 : 10;   // (loads in flight; one batch on 152 SMs)
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p0 = grp; p0 < G; p0 += GG * BATCH) {
            float4 v[BATCH];
#pragma unroll
            for (int k = 0; k < BATCH; ++k) {
                const int p = p0 + k * GG;
                v[k] = p < G ? __ldcg(gp + (size_t)p * (S::N / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < BATCH; ++k) {
                s.x += v[k].x; s.y += v[k].y; s.z += v[k].z; s.w += v[k].w;
            }
        }
        sgs[grp * GC + col] = s;
    }
    __syncthreads();
    if (tid < GC) {
        float4 t = sgs[tid];
#pragma unroll
        for (int k = 1; k < GG; ++k) {
            const float4 v = sgs[k * GC + tid];
            t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
        }
        LOOP_AT(float4, S::O_G)[tid] = t;
    }
    __syncthreads();
}

template <class S>
__device__ __forceinline__ void loop_begin(const LoopArgs& q)
{
    LOOP_SMEM;
    constexpr int NN = S::NN, N = S::N, WL = S::WL, THREADS = S::THREADS;
    const int tid = fresh_tid(), blk = blockIdx.x, r0 = 2 * blk;
    const int i0 = (int)(((long long)q.m * blk) / gridDim.x);
    const int nrows = (int)(((long long)q.m * (blk + 1)) / gridDim.x) - i0;
    LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    if (tid == 0) {
        st->gave_up = st->end = 0;
        st->pending = q.ctrl->pending;
        st->algo = q.ctrl->algo;
        st->i0 = i0;
        st->nrows = nrows;
        st->tol = q.ctrl->tol;
    }
    if constexpr (S::RREG == 0) if (tid == 0) {
        uint64_t* full = LOOP_AT(uint64_t, S::O_BAR);
        for (int s = 0; s < S::NPC; ++s) mbar_init(&full[s], 1);
        fence_mbar_init();
        Ring& g = *LOOP_AT(Ring, S::O_RING);
        g.p0 = q.P0 + (size_t)i0 * N * S::B0;
        g.p1 = S::B1 > 0 ? q.P1 + (size_t)i0 * N * S::B1 : nullptr;
        g.pol = l2_policy_evict_first();
        g.nrows = nrows;
        g.pieces = (nrows + S::RP - 1) / S::RP;
        const bool resident = g.pieces <= S::NPC;
        g.passes = nrows == 0 ? 0 : resident ? 1 : q.iters;
        g.pass = g.o = g.slot = g.phase = 0;
        for (int k = 0; k < S::NPC; ++k) ring_issue<S>();
    }
    if (nrows <= S::YMAX) {
        for (int i = tid; i < nrows; i += THREADS) LOOP_AT(float, S::O_Y)[i] = q.y[i0 + i];
        if constexpr (S::PREC == 2)
            for (int i = tid; i < nrows; i += THREADS) LOOP_AT(float, S::O_S)[i] = q.rscale[i0 + i];
    }
    if (blk < S::NP) {
        float* su = LOOP_AT(float, S::O_SU);
        float* swl = LOOP_AT(float, S::O_WL);
        float* rdiv = LOOP_AT(float, S::O_RD);
        const int par = q.ctrl->wpar;
        for (int i = tid; i < NN; i += THREADS) {
            LOOP_AT(float2, S::O_TW)[i] = q.tw[i];
            rdiv[i] = 1.0f / solve_divisor(q.s2, i, blk, q.beta, q.mu_over_tau);
            rdiv[NN + i] = 1.0f / solve_divisor(q.s2, i, NN / 2, q.beta, q.mu_over_tau);
        }
        for (int i = tid; i < 4 * NN; i += THREADS) {
            const int rr = i / NN, c = i - rr * NN;
            su[i] = q.u[((r0 - 1 + rr + NN) % NN) * NN + c];
        }
        for (int i = tid; i < WL; i += THREADS) {
            const int rr = i / NN, c = i - rr * NN;
            const size_t gi = (size_t)par * 2 * N + ((r0 - 1 + rr + NN) % NN) * NN + c;
            swl[i] = q.w[gi];
            swl[WL + i] = q.w[gi + N];
            swl[2 * WL + i] = q.lam[gi];
            swl[3 * WL + i] = q.lam[gi + N];
        }
        for (int i = tid; i < 2 * NN; i += THREADS) LOOP_AT(float, S::O_G)[i] = q.g[r0 * NN + i];
    }
    __syncthreads();
    if (blk < S::NP) loop_shrink<S>(q.beta, 0, tid, THREADS);
    __syncthreads();
}

// End of the run after iteration `it`: the u-step's blocks write u, w, lambda and g of their
// rows (w and lambda to the copy they came from), block 0 the control block.
template <class S>
__device__ __forceinline__ void loop_end(const LoopArgs& q, int it)
{
    LOOP_SMEM;
    constexpr int NN = S::NN, N = S::N, WL = S::WL;
    const int tid = fresh_tid(), blk = blockIdx.x, r0 = 2 * blk;
    LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    Ctrl* ctrl = q.ctrl;
    if (__syncthreads_or(st->gave_up)) {
        if (tid == 0) set_error(ctrl, ERR_TIMEOUT);
    } else if (blk < S::NP) {
        const float* su = LOOP_AT(float, S::O_SU);
        const float* src = LOOP_AT(float, S::O_WL) + (it & 1) * 4 * WL;
        const int par = ctrl->wpar;
        for (int i = tid; i < 2 * NN; i += S::THREADS) {
            const size_t gi = (size_t)r0 * NN + i, wi = (size_t)par * 2 * N + gi;
            q.u[gi] = su[NN + i];
            q.g[gi] = LOOP_AT(float, S::O_G)[i];
            q.w[wi] = src[NN + i];
            q.w[wi + N] = src[WL + NN + i];
            q.lam[wi] = src[2 * WL + NN + i];
            q.lam[wi + N] = src[3 * WL + NN + i];
        }
    }
    bool ends = blk == 0;   // this block writes the control block
    if constexpr (S::RREG > 0) {   // r of the block's rows and its norm; the last block to come adds the norms
        const float* sr = LOOP_AT(float, S::O_R);
        float2 v = make_float2(0.f, 0.f);
        for (int i = tid; i < st->nrows; i += S::THREADS) {
            q.r[st->i0 + i] = sr[i];
            v = ds_add(v, ds_sq(sr[i]));
        }
        v = block_sum_ds(v, LOOP_AT(float2, S::O_DRED));
        if (tid == 0) q.r2part[blk] = v;
        ends = last_block_all(&ctrl->ticket_gather, &st->last);
    }
    if (!__syncthreads_or(st->gave_up)) {
        if (ends) {
            // ||r||^2 = sum of the G partials, fixed order (every partial is visible: the
            // arrivals of this iteration were awaited, or this block is the last)
            float2* dred = LOOP_AT(float2, S::O_DRED);
            float2 v = make_float2(0.f, 0.f);
            for (int p = tid; p < (int)gridDim.x; p += S::THREADS) v = ds_add(v, __ldcg(q.r2part + p));
            v = warp_sum_ds(v);
            if ((tid & 31) == 0) dred[tid >> 5] = v;
            __syncthreads();
            if (tid == 0) {
                float2 t = dred[0];
                for (int w = 1; w < S::WARPS; ++w) t = ds_add(t, dred[w]);
                ctrl->r2 = ds_value(t);
                ctrl->it = it;
                ctrl->done = 1;
                ctrl->du2 = st->du2;
                ctrl->u2 = st->u2;
                if (st->algo == 0) ctrl->pending = 1;   // u moved: its multiplier update is due
                if (st->end == 2) ctrl->stop_by_tol = 1;
                if (st->end == 3) set_error(ctrl, ERR_NONFINITE);
            }
        }
    }
    if constexpr (S::RREG == 0) if (tid == 0) {   // let the copies still in flight land (bounded): every slot's last phase
        const Ring& g = *LOOP_AT(Ring, S::O_RING);
        const int used = g.passes == 1 ? min(S::NPC, g.pieces) : g.passes > 1 ? S::NPC : 0;
        uint64_t* full = LOOP_AT(uint64_t, S::O_BAR);
        for (int s = 0; s < used; ++s)
            mbar_wait(&full[s], (uint32_t)(s < g.slot ? g.phase : g.phase ^ 1), drain_budget(q.budget));
    }
}

}  // namespace

template <int NN, int PREC, int TC, int VW, int V, int RL, int RB, int RP, int NPC>
__global__ void __maxnreg__(128) k_loop(const __grid_constant__ LoopArgs q)
{
    using S = LoopShape<NN, PREC, TC, VW, V, RL, RB, RP, NPC>;
    LOOP_SMEM;
    volatile LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    loop_begin<S>(q);
    int it = 0;
    while (true) {
        ++it;
        if (blockIdx.x < S::NP && threadIdx.x < 32) loop_ustep<S>(q, it);
        loop_pass<S>(q, it);
        __syncthreads();
        loop_arrive<S>(q, it);
        // (the vote makes the outcome the same for every thread of the block)
        if (__syncthreads_or(st->gave_up)) break;
        const int end = st->end;
        if (blockIdx.x < S::NP) loop_gather<S>(q);
        if (end) break;
    }
    loop_end<S>(q, it);
}

template <int NN, int TC, int V, int RL, int RREG>
__global__ void __launch_bounds__(TC * RL, 1) k_loop_reg(const __grid_constant__ LoopArgs q)
{
    using S = RegShape<NN, TC, V, RL, RREG>;
    LOOP_SMEM;
    volatile LoopState* st = LOOP_AT(LoopState, S::O_STATE);
    loop_begin<S>(q);
    uint64_t a[RREG][S::CP];
    const int lane_row = threadIdx.x / TC;
    reg_load_rows<S>(q, st->i0, st->nrows, lane_row, threadIdx.x - lane_row * TC, a, LOOP_AT(float, S::O_A));
    __syncthreads();
    int it = 0;
    while (true) {
        ++it;
        if (blockIdx.x < S::NP && threadIdx.x < 32) loop_ustep<S>(q, it);
        loop_pass_reg<S>(q, it, a);
        __syncthreads();
        loop_arrive<S>(q, it);
        if (__syncthreads_or(st->gave_up)) break;
        const int end = st->end;
        if (blockIdx.x < S::NP) loop_gather<S>(q);
        if (end) break;
    }
    loop_end<S>(q, it);
}

// ---------------------------------------------------------------------------
// Shape table: (precision, n) -> (TC, VW, V, RL, RB, RP, NPC), rows a block takes at least.
// The blocks are at least the n/2 of the u-step and at most one per SM.
// (Up to 64 x 64 only what does not fit on chip comes here: on 152 SMs m > 3192 at n = 64, 4712 at
// 48, 9272 at 32, 37544 at 16.)
// ---------------------------------------------------------------------------
//    precision, n, minimum rows per block, TC, VW, V, RL, RB, RP, NPC
#define TVCS_LOOP_TABLE(X)                   \
    X(0, 16, 8, 64, 4, 1, 8, 2, 16, 4)       \
    X(0, 32, 8, 256, 4, 1, 2, 4, 8, 4)       \
    X(0, 48, 4, 384, 2, 3, 1, 4, 4, 4)       \
    X(0, 64, 4, 512, 4, 2, 1, 4, 4, 3)       \
    X(0, 96, 1, 512, 2, 9, 1, 2, 1, 5)       \
    X(1, 32, 8, 256, 4, 1, 2, 4, 8, 4)       \
    X(1, 64, 4, 512, 8, 1, 1, 4, 4, 3)       \
    X(2, 32, 8, 256, 4, 1, 2, 4, 8, 4)       \
    X(2, 64, 4, 512, 8, 1, 1, 4, 4, 4)

template <int NN, int PREC, int TC, int VW, int V, int RL, int RB, int RP, int NPC>
static bool loop_configure_t()
{
    using S = LoopShape<NN, PREC, TC, VW, V, RL, RB, RP, NPC>;
    auto kernel = k_loop<NN, PREC, TC, VW, V, RL, RB, RP, NPC>;
    int per = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, S::THREADS, S::SMEM) != cudaSuccess ||
        per < 1) {
        cudaGetLastError();
        return false;
    }
    return true;
}

bool loop_configure(int prec, int n)
{
#define X(PR, NN, MR, TC, VW, V, RL, RB, RP, NPC) \
    if (prec == PR && n == NN) return loop_configure_t<NN, PR, TC, VW, V, RL, RB, RP, NPC>();
    TVCS_LOOP_TABLE(X)
#undef X
    return false;
}

int loop_grid(int prec, int n, int m, int num_sms)
{
    int mr = 0;
#define X(PR, NN, MR, TC, VW, V, RL, RB, RP, NPC) \
    if (prec == PR && n == NN) mr = MR;
    TVCS_LOOP_TABLE(X)
#undef X
    if (mr == 0 || num_sms < n / 2) return 0;
    return std::min(num_sms, std::max(n / 2, (m + mr - 1) / mr));
}

template <int NN, int PREC, int TC, int VW, int V, int RL, int RB, int RP, int NPC>
static cudaError_t launch_loop_t(int grid, const LoopArgs& a, cudaStream_t s)
{
    using S = LoopShape<NN, PREC, TC, VW, V, RL, RB, RP, NPC>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(S::THREADS, 1, 1);
    cfg.dynamicSmemBytes = S::SMEM;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // the blocks wait for one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_loop<NN, PREC, TC, VW, V, RL, RB, RP, NPC>, a);
}

// ---------------------------------------------------------------------------
// Shapes with every row on chip: n -> (rows per block aimed at, TC, V, RL, RREG).  Fewer threads
// with more columns each leave the registers for A (8 rows of 16 columns at n = 64).  Measured
// at n = 64, m = 1229: 256 x 16 columns 9.7 us, 512 x 8 9.6; n = 48: 288 x 8 8.0, 139 blocks of 5
// rows instead of 87 9.0; n = 32: 39 blocks of 8 rows 7.3, 20 of 16 8.1.
// ---------------------------------------------------------------------------
#define TVCS_REG_TABLE(X)     \
    X(16, 32, 64, 1, 4, 8)    \
    X(32, 8, 256, 1, 1, 8)    \
    X(48, 8, 288, 2, 1, 8)    \
    X(64, 8, 256, 4, 1, 8)

template <int NN, int TC, int V, int RL, int RREG>
static bool reg_configure_t()
{
    using S = RegShape<NN, TC, V, RL, RREG>;
    auto kernel = k_loop_reg<NN, TC, V, RL, RREG>;
    int per = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem(S::RMAX)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, S::THREADS, S::smem(S::RMAX)) != cudaSuccess ||
        per < 1) {
        cudaGetLastError();
        return false;
    }
    return true;
}

bool reg_configure(int n)
{
#define X(NN, MR, TC, V, RL, RREG) \
    if (n == NN) return reg_configure_t<NN, TC, V, RL, RREG>();
    TVCS_REG_TABLE(X)
#undef X
    return false;
}

int reg_grid(int n, int m, int num_sms)
{
    if (num_sms < n / 2) return 0;
#define X(NN, MR, TC, V, RL, RREG)                                              \
    if (n == NN) {                                                              \
        const int g = std::min(num_sms, std::max(n / 2, (m + MR - 1) / MR));    \
        return (m + g - 1) / g <= RegShape<NN, TC, V, RL, RREG>::RMAX ? g : 0;  \
    }
    TVCS_REG_TABLE(X)
#undef X
    return 0;
}

cudaError_t launch_loop_reg(int n, int grid, const LoopArgs& a, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // the blocks wait for one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#define X(NN, MR, TC, V, RL, RREG)                                                    \
    if (n == NN) {                                                                    \
        using S = RegShape<NN, TC, V, RL, RREG>;                                      \
        cfg.blockDim = dim3(S::THREADS, 1, 1);                                        \
        cfg.dynamicSmemBytes = S::smem((a.m + grid - 1) / grid);                      \
        return cudaLaunchKernelEx(&cfg, k_loop_reg<NN, TC, V, RL, RREG>, a);          \
    }
    TVCS_REG_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t launch_loop(int prec, int n, int grid, const LoopArgs& a, cudaStream_t s)
{
#define X(PR, NN, MR, TC, VW, V, RL, RB, RP, NPC) \
    if (prec == PR && n == NN) return launch_loop_t<NN, PR, TC, VW, V, RL, RB, RP, NPC>(grid, a, s);
    TVCS_LOOP_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace tvcs
