// The whole iteration loop with the partial-DCT encoder (Sec. 3.2; reading C18) as ONE
// launch of one thread-block cluster: rows a1-a7 of every iteration and eq. (stop), for
// A u = (C U C^T)[rows] with C the orthonormal n x n DCT-II matrix.
//
// Block q of the cluster owns image rows [q R, (q+1) R), R = n / CL, the DCT columns of the
// same indices and QC = n / 2 / CL column slots of the half spectrum (slot 0: the two real
// columns 0 and n/2 as one complex column).  All transforms are length-n complex FFTs, one
// by one warp: a DCT-II of two real sequences is the FFT of the even entries followed by the
// odd ones reversed (J. Makhoul, IEEE Trans. ASSP 28, 1980), both sequences packed as real
// and imaginary part, and a rotation by exp(-i pi k / 2n); the transposed transform runs the
// steps backwards.  An iteration is eight such phases and four cluster barriers:
//   1  row DCTs of u -> coefficients to the blocks of their columns       | norms of eq. (stop)
//   2  column DCTs, r at the sampled positions, S, column transforms back |
//      -> to the blocks of their rows                                     | w-step, D^T y
//   3  row transforms back (g), right-hand side, row FFTs -> column slots |
//   4  column FFTs, divide, inverse -> rows;  inverse row FFTs, u += d    |
// (left: R/2 warps, one pair of rows or columns each; right: the other four warps
// meanwhile).  Values go straight into the owner's shared memory.
//
// What bounds it: the latency of the four cluster barriers and of the eight transforms (three
// shared-memory stages each); the arithmetic is 2.6 MFLOP an iteration at n = 128.  The
// chain that it replaces ran two clusters of 16 SMs (u-solve; four dense n x n transforms
// with two whole matrices exchanged through L2) with two kernel boundaries: 18.7 us an
// iteration at n = 128, here 9.7 (300 iterations with the start point and the end of the run
// 5.72 -> 2.97 ms; the image's error against binary64, mean of six inputs, 3.1e-7 -> 2.3e-7).
#include <cooperative_groups.h>

#include "common.cuh"
#include "fft.cuh"
#include "kernels.h"
#include "usolve_steps.cuh"

namespace cg = cooperative_groups;

namespace tvcs {

namespace {

constexpr int DL_THREADS = 256;   // 4 warps of transforms, 4 helpers
constexpr int DL_HELP = 128;      // threads of the helpers

template <int NN, int CL>
struct DctLoopShape {
    static constexpr int R = NN / CL, PAIRS = R / 2, QC = NN / 2 / CL, NP = NN / 2;
    static constexpr int N = NN * NN, WL = (R + 1) * NN;
    static_assert(NN % CL == 0 && R % 2 == 0 && NP % CL == 0 && PAIRS <= 4 && QC <= 4 && CL <= 16, "split");
    static constexpr size_t O_TW = 0;                          // exp(2 pi i t / n)
    static constexpr size_t O_IC = O_TW + NN * 8;              // s_k exp(i pi k / 2n)
    static constexpr size_t O_RD = O_IC + NN * 8;              // reciprocal divisors of the slots and of column n/2
    static constexpr size_t O_SU = O_RD + (QC + 1) * NN * 4;   // u rows r0-1 .. r0+R
    static constexpr size_t O_WL = O_SU + (R + 2) * NN * 4;    // w1, w2, l1, l2 of rows r0-1 .. r0+R-1
    static constexpr size_t O_Y1 = O_WL + 4 * WL * 4;
    static constexpr size_t O_Y2 = O_Y1 + R * NN * 4;
    static constexpr size_t O_DTY = O_Y2 + (R + 1) * NN * 4;   // [PAIRS][n] D^T y of two rows
    static constexpr size_t O_COL = O_DTY + PAIRS * NN * 8;    // [R][n] row coefficients by column, cluster-written
    static constexpr size_t O_ROW = O_COL + R * NN * 4;        // [R][n] column-transformed back, cluster-written
    static constexpr size_t O_FCOL = O_ROW + R * NN * 4;       // [QC][n] complex, cluster-written
    static constexpr size_t O_SPEC = O_FCOL + QC * NN * 8;     // [R][n/2] complex, cluster-written
    static constexpr size_t O_FA = O_SPEC + R * NP * 8;        // per transform warp: two buffers of n complex
    static constexpr size_t O_FB = O_FA + 4 * NN * 8;
    static constexpr size_t O_Z = O_FB + 4 * NN * 8;           // [PAIRS][n] the last step n^2 d, packed rows
    static constexpr size_t O_S = O_Z + PAIRS * NN * 8;        // per transform warp: two real sequences
    static constexpr size_t O_G = O_S + 4 * 2 * NN * 4;        // [R][n] g
    static constexpr size_t O_POS = O_G + R * NN * 4;          // [R][n] position of the coefficient in r, or -1
    static constexpr size_t O_F = O_POS + R * NN * 4;          // [R][n] its measurement
    static constexpr size_t O_NORM = ((O_F + R * NN * 4 + 15) / 16) * 16;   // [CL][4] float4: du2, u2 per pair
    static constexpr size_t O_RED = O_NORM + CL * 4 * 16;      // [64] float2, then [CL] float2 of rank 0
    static constexpr size_t O_END = O_RED + (64 + 16) * 8;     // [4] int
    static constexpr size_t SMEM = O_END + 16;
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Place of entry t of the reordered sequence (evens, then odds reversed).
template <int NN>
__device__ __forceinline__ int dct_place(int t)
{
    return 2 * t < NN ? 2 * t : 2 * NN - 1 - 2 * t;
}

// DCT-II coefficients k of the two sequences packed in Z (its FFT): (first, second).
template <int NN>
__device__ __forceinline__ float2 dct_coef(const float2* Z, const float2* ic, int k)
{
    const float2 z = Z[k];
    const float2 c = ic[k];
    if (k == 0) return make_float2(c.x * z.x, c.x * z.y);
    const float2 y = Z[NN - k];
    return make_float2(c.x * (z.x + y.x) + c.y * (z.y - y.y), c.x * (z.y + y.y) - c.y * (z.x - y.x));
}

// Entry k of the packed spectrum whose inverse FFT is the reordered transposed transform of
// the coefficient sequences a and b.
template <int NN>
__device__ __forceinline__ float2 dct_back(const float* a, const float* b, const float2* ic, int k)
{
    const float2 c = ic[k];
    if (k == 0) return make_float2(c.x * a[0], c.x * b[0]);
    const float ak = a[k], an = a[NN - k], bk = b[k], bn = b[NN - k];
    const float v1x = c.x * ak + c.y * an, v1y = c.y * ak - c.x * an;
    const float v2x = c.x * bk + c.y * bn, v2y = c.y * bk - c.x * bn;
    return make_float2(v1x - v2y, v1y + v2x);
}

}  // namespace

template <int NN, int CL>
__global__ void __launch_bounds__(DL_THREADS, 1) k_dct_loop(const __grid_constant__ DctLoopArgs q)
{
    using S = DctLoopShape<NN, CL>;
    constexpr int R = S::R, PAIRS = S::PAIRS, QC = S::QC, NP = S::NP, N = S::N, WL = S::WL;
    extern __shared__ __align__(16) unsigned char smem[];
    float2* tw = reinterpret_cast<float2*>(smem + S::O_TW);
    float2* ic = reinterpret_cast<float2*>(smem + S::O_IC);
    float* rdiv = reinterpret_cast<float*>(smem + S::O_RD);
    float* su = reinterpret_cast<float*>(smem + S::O_SU);
    float* swl = reinterpret_cast<float*>(smem + S::O_WL);
    float* sy1 = reinterpret_cast<float*>(smem + S::O_Y1);
    float* sy2 = reinterpret_cast<float*>(smem + S::O_Y2);
    float2* dty = reinterpret_cast<float2*>(smem + S::O_DTY);
    float* colb = reinterpret_cast<float*>(smem + S::O_COL);
    float* rowb = reinterpret_cast<float*>(smem + S::O_ROW);
    float2* fcol = reinterpret_cast<float2*>(smem + S::O_FCOL);
    float2* spec = reinterpret_cast<float2*>(smem + S::O_SPEC);
    float2* zbuf = reinterpret_cast<float2*>(smem + S::O_Z);
    float* sg = reinterpret_cast<float*>(smem + S::O_G);
    int* pos = reinterpret_cast<int*>(smem + S::O_POS);
    float* fv = reinterpret_cast<float*>(smem + S::O_F);
    float4* norms = reinterpret_cast<float4*>(smem + S::O_NORM);
    float2* red = reinterpret_cast<float2*>(smem + S::O_RED);
    int* send = reinterpret_cast<int*>(smem + S::O_END);

    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = rank * R;
    float2* fa = reinterpret_cast<float2*>(smem + S::O_FA) + (warp & 3) * NN;
    float2* fb = reinterpret_cast<float2*>(smem + S::O_FB) + (warp & 3) * NN;
    float* sa = reinterpret_cast<float*>(smem + S::O_S) + (warp & 3) * 2 * NN;
    float* sb = sa + NN;
    Ctrl* ctrl = q.ctrl;
    const int algo = ctrl->algo, par = ctrl->wpar;
    const double tol = ctrl->tol;
    int pending = ctrl->pending;

    // ---------------- state ----------------
    for (int i = tid; i < NN; i += DL_THREADS) {
        tw[i] = q.tw[i];
        ic[i] = q.ic[i];
    }
    for (int i = tid; i < (QC + 1) * NN; i += DL_THREADS) {
        const int f = i / NN, p = i - f * NN;
        rdiv[i] = 1.0f / solve_divisor(q.s2, p, f < QC ? rank * QC + f : NP, q.beta, q.mu_over_tau);
    }
    for (int i = tid; i < (R + 2) * NN; i += DL_THREADS) {
        const int rr = i / NN, c = i - rr * NN;
        su[i] = q.u[((r0 - 1 + rr + NN) % NN) * NN + c];
    }
    for (int i = tid; i < WL; i += DL_THREADS) {
        const int rr = i / NN, c = i - rr * NN;
        const size_t gi = (size_t)par * 2 * N + ((r0 - 1 + rr + NN) % NN) * NN + c;
        swl[i] = q.w[gi];
        swl[WL + i] = q.w[gi + N];
        swl[2 * WL + i] = q.lam[gi];
        swl[3 * WL + i] = q.lam[gi + N];
    }
    for (int i = tid; i < R * NN; i += DL_THREADS) {   // columns r0 .. r0+R-1 of the coefficients
        const int p = q.pos[(size_t)r0 * NN + i];
        pos[i] = p;
        fv[i] = p >= 0 ? q.y[p] : 0.f;
    }
    const float beta = q.beta, inv_beta = 1.0f / q.beta, mu = q.mu;
    const float sc = 1.0f / (float)N;
    float2 r2 = make_float2(0.f, 0.f);   // double-single ||r||^2 of this lane's coefficients
    int it = 0, end = 0;
    cluster.sync();   // every block has started and read its state

    while (true) {
        // ---------------- 1: row DCTs of u; norms of the last step ----------------
        if (warp < PAIRS) {
            const int lr = 2 * warp;
            const float *ua = su + (lr + 1) * NN, *ub = ua + NN;
            for (int t = lane; t < NN; t += 32) {
                const int c = dct_place<NN>(t);
                fa[t] = make_float2(ua[c], ub[c]);
            }
            __syncwarp();
            const float2* Z = fft_warp<NN, false>(fa, fb, tw, lane);
            for (int k = lane; k < NN; k += 32) {
                float* dst = cluster.map_shared_rank(colb, k / R) + (k % R) * NN + r0 + lr;
                *reinterpret_cast<float2*>(dst) = dct_coef<NN>(Z, ic, k);
            }
            // halo rows for the neighbours' w-step
            if (warp == 0) {
                float* dst = cluster.map_shared_rank(su, (rank + CL - 1) % CL) + (R + 1) * NN;
                for (int c = lane; c < NN; c += 32) dst[c] = su[NN + c];
            }
            if (warp == PAIRS - 1) {
                float* dst = cluster.map_shared_rank(su, (rank + 1) % CL);
                for (int c = lane; c < NN; c += 32) dst[c] = su[R * NN + c];
            }
        } else if (warp >= 4 && warp - 4 < PAIRS && it > 0) {
            // ||d||^2 and ||u||^2 (before the step) of one pair of rows, to every block
            const int pr = warp - 4;
            const float2* z = zbuf + pr * NN;
            float2 du2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
            for (int c = lane; c < NN; c += 32) {
                const float2 v = z[c];
                du2 = ds_add(du2, ds_sq(v.x * sc));
                du2 = ds_add(du2, ds_sq(v.y * sc));
                u2 = ds_add(u2, ds_sq(sg[2 * pr * NN + c]));
                u2 = ds_add(u2, ds_sq(sg[(2 * pr + 1) * NN + c]));
            }
            du2 = warp_sum_ds(du2);
            u2 = warp_sum_ds(u2);
            if (lane < CL) cluster.map_shared_rank(norms, lane)[rank * 4 + pr] = make_float4(du2.x, du2.y, u2.x, u2.y);
        }
        cluster.sync();

        // ---------------- eq. (stop) for iteration `it` (the same in every block) ----------------
        if (warp >= 4) {
            if (warp == 4) {
                int e = 0;
                if (it > 0) {
                    float2 du2 = make_float2(0.f, 0.f), u2 = make_float2(0.f, 0.f);
                    for (int j = lane; j < CL * PAIRS; j += 32) {
                        const float4 v = norms[(j / PAIRS) * 4 + j % PAIRS];
                        du2 = ds_add(du2, make_float2(v.x, v.y));
                        u2 = ds_add(u2, make_float2(v.z, v.w));
                    }
                    du2 = warp_sum_ds(du2);
                    u2 = warp_sum_ds(u2);
                    const double tdu = ds_value(du2), tu = ds_value(u2);
                    e = it >= q.iters ? 1 : 0;
                    if (!isfinite(tdu) || !isfinite(tu))
                        e = 3;
                    else if (tol > 0.0 && (tu > 0.0 ? tdu <= tol * tol * tu : tdu == 0.0))
                        e = 2;   // eq. (stop), reading C5
                    if (lane == 0 && rank == 0) {
                        ctrl->du2 = tdu;
                        ctrl->u2 = tu;
                    }
                }
                if (lane == 0) send[0] = e;
            }
            named_barrier(1, DL_HELP);
            // ---------------- w-step and D^T y (a1-a3) ----------------
            if (send[0] == 0) {
                for (int i = tid - DL_HELP; i < WL; i += DL_HELP) {
                    const int rr = i / NN, c = i - rr * NN;
                    const int cp = (c + 1 == NN) ? 0 : c + 1;
                    const float uc = su[i];
                    const float d1 = su[rr * NN + cp] - uc, d2 = su[i + NN] - uc;
                    float l1 = swl[2 * WL + i], l2 = swl[3 * WL + i];
                    if (pending) {   // eq. (udlamb) for the previous iteration
                        l1 -= beta * (swl[i] - d1);
                        l2 -= beta * (swl[WL + i] - d2);
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
                    swl[i] = w1;
                    swl[WL + i] = w2;
                    swl[2 * WL + i] = l1;
                    swl[3 * WL + i] = l2;
                }
                named_barrier(1, DL_HELP);
                step_dty<NN>(sy1, sy2, R, dty, tid - DL_HELP, DL_HELP);
            }
        }
        // ---------------- 2: column DCTs, r, columns back ----------------
        else if (warp < PAIRS) {
            const int c0 = 2 * warp;   // local columns c0, c0 + 1
            for (int t = lane; t < NN; t += 32) {
                const int i = dct_place<NN>(t);
                fa[t] = make_float2(colb[c0 * NN + i], colb[(c0 + 1) * NN + i]);
            }
            __syncwarp();
            const float2* Z = fft_warp<NN, false>(fa, fb, tw, lane);
            r2 = make_float2(0.f, 0.f);
            for (int k = lane; k < NN; k += 32) {
                const float2 x = dct_coef<NN>(Z, ic, k);
                float s0 = 0.f, s1 = 0.f;
                const int p0 = pos[c0 * NN + k], p1 = pos[(c0 + 1) * NN + k];
                if (p0 >= 0) {
                    s0 = x.x - fv[c0 * NN + k];
                    q.r[p0] = s0;
                    r2 = ds_add(r2, ds_sq(s0));
                }
                if (p1 >= 0) {
                    s1 = x.y - fv[(c0 + 1) * NN + k];
                    q.r[p1] = s1;
                    r2 = ds_add(r2, ds_sq(s1));
                }
                sa[k] = s0;
                sb[k] = s1;
            }
            __syncwarp();
            for (int k = lane; k < NN; k += 32) fa[k] = dct_back<NN>(sa, sb, ic, k);
            __syncwarp();
            const float2* z = fft_warp<NN, true>(fa, fb, tw, lane);
            for (int t = lane; t < NN; t += 32) {
                const int i = dct_place<NN>(t);
                float* dst = cluster.map_shared_rank(rowb, i / R) + (i % R) * NN + r0 + c0;
                *reinterpret_cast<float2*>(dst) = z[t];
            }
        }
        cluster.sync();
        end = send[0];

        // ---------------- 3: rows back (g), right-hand side, row FFTs ----------------
        if (warp < PAIRS) {
            const int lr = 2 * warp;
            const float *ra = rowb + lr * NN, *rb = ra + NN;
            for (int k = lane; k < NN; k += 32) fa[k] = dct_back<NN>(ra, rb, ic, k);
            __syncwarp();
            const float2* z = fft_warp<NN, true>(fa, fb, tw, lane);
            if (end) {
                for (int t = lane; t < NN; t += 32) {
                    const int c = dct_place<NN>(t);
                    sg[lr * NN + c] = z[t].x;
                    sg[(lr + 1) * NN + c] = z[t].y;
                }
            } else {
                float2* wa = z == fa ? fb : fa;
                for (int t = lane; t < NN; t += 32) {
                    const int c = dct_place<NN>(t);
                    const float2 d = dty[warp * NN + c], g = z[t];
                    wa[c] = make_float2(d.x - mu * g.x, d.y - mu * g.y);
                }
                __syncwarp();
                const float2* Z = fft_warp<NN, false>(wa, wa == fa ? fb : fa, tw, lane);
                // the half spectra of the two rows to the blocks of their column slots
                for (int s = lane; s < NP; s += 32) {
                    const float2 a = Z[s], b = Z[(NN - s) % NN];
                    float2* dst = cluster.map_shared_rank(fcol, s / QC) + (s % QC) * NN + r0 + lr;
                    if (s == 0) {
                        const float2 n2 = Z[NP];
                        dst[0] = make_float2(a.x, n2.x);
                        dst[1] = make_float2(a.y, n2.y);
                    } else {
                        dst[0] = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
                        dst[1] = make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x));
                    }
                }
            }
        }
        if (end) break;
        cluster.sync();

        // ---------------- 4: column slots ----------------
        if (warp < QC) {
            float2* X = fft_warp<NN, false>(fcol + warp * NN, fb, tw, lane);
            const float* rd = rdiv + warp * NN;
            if (rank != 0 || warp != 0) {
                for (int p = lane; p < NN; p += 32) X[p] = make_float2(X[p].x * rd[p], X[p].y * rd[p]);
            } else {   // columns 0 and n/2, separated by conjugate symmetry
                for (int k = lane; 2 * k <= NN; k += 32) {
                    const int km = (NN - k) % NN;
                    const float2 zk = X[k], zm = X[km];
                    const float a0 = rdiv[k], an = rdiv[QC * NN + k];
                    const float2 e0 = make_float2(0.5f * (zk.x + zm.x) * a0, 0.5f * (zk.y - zm.y) * a0);
                    const float2 en = make_float2(0.5f * (zk.y + zm.y) * an, -0.5f * (zk.x - zm.x) * an);
                    X[k] = make_float2(e0.x - en.y, e0.y + en.x);
                    if (km != k) X[km] = make_float2(e0.x + en.y, en.x - e0.y);
                }
            }
            __syncwarp();
            const float2* Y = fft_warp<NN, true>(X, X == fb ? fa : fb, tw, lane);
            for (int p = lane; p < NN; p += 32)
                cluster.map_shared_rank(spec, p / R)[(p % R) * NP + rank * QC + warp] = Y[p];
        }
        cluster.sync();

        // ---------------- inverse rows, u <- u + d ----------------
        if (warp < PAIRS) {
            const int lr = 2 * warp;
            for (int s = lane; s < NP; s += 32) {
                const float2 Xv = spec[lr * NP + s], Yv = spec[(lr + 1) * NP + s];
                if (s == 0) {
                    fa[0] = make_float2(Xv.x, Yv.x);
                    fa[NP] = make_float2(Xv.y, Yv.y);
                } else {
                    fa[s] = make_float2(Xv.x - Yv.y, Xv.y + Yv.x);
                    fa[NN - s] = make_float2(Xv.x + Yv.y, Yv.x - Xv.y);
                }
            }
            __syncwarp();
            const float2* z = fft_warp<NN, true>(fa, fb, tw, lane);
            float *ua = su + (lr + 1) * NN, *ub = ua + NN;
            for (int c = lane; c < NN; c += 32) {
                const float2 v = z[c];
                const float oa = ua[c], ob = ub[c];
                zbuf[warp * NN + c] = v;
                sg[lr * NN + c] = oa;   // the old u, for the norms
                sg[(lr + 1) * NN + c] = ob;
                ua[c] = oa + v.x * sc;
                ub[c] = ob + v.y * sc;
            }
        }
        ++it;
        pending = algo == 0 ? 1 : 0;
        __syncthreads();
    }

    // ---------------- end of the run ----------------
    r2 = warp < PAIRS ? r2 : make_float2(0.f, 0.f);
    r2 = block_sum_ds(r2, red);   // (barriers: sg is complete as well)
    if (tid == 0) cluster.map_shared_rank(red, 0)[64 + rank] = r2;
    for (int i = tid; i < R * NN; i += DL_THREADS) {
        const size_t gi = (size_t)r0 * NN + i, wi = (size_t)par * 2 * N + gi;
        q.u[gi] = su[NN + i];
        q.g[gi] = sg[i];
        q.w[wi] = swl[NN + i];
        q.w[wi + N] = swl[WL + NN + i];
        q.lam[wi] = swl[2 * WL + NN + i];
        q.lam[wi + N] = swl[3 * WL + NN + i];
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        float2 t = red[64];
        for (int k = 1; k < CL; ++k) t = ds_add(t, red[64 + k]);
        ctrl->r2 = ds_value(t);
        ctrl->it = it;
        ctrl->done = 1;
        if (algo == 0) ctrl->pending = 1;   // u moved: its multiplier update is due
        if (end == 2) ctrl->stop_by_tol = 1;
        if (end == 3) set_error(ctrl, ERR_NONFINITE);
    }
}

// ---------------------------------------------------------------------------
// Host side.  n -> blocks of the cluster.
// ---------------------------------------------------------------------------
#define TVCS_DCT_LOOP_TABLE(X) X(16, 8) X(32, 16) X(48, 8) X(64, 16) X(96, 16) X(128, 16)

template <int NN, int CL>
static cudaLaunchConfig_t dct_loop_config(cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL, 1, 1);
    cfg.blockDim = dim3(DL_THREADS, 1, 1);
    cfg.dynamicSmemBytes = DctLoopShape<NN, CL>::SMEM;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = CL;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <int NN, int CL>
static bool dct_loop_configure_t()
{
    auto kernel = k_dct_loop<NN, CL>;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = dct_loop_config<NN, CL>(&attr);
    int clusters = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)DctLoopShape<NN, CL>::SMEM) != cudaSuccess ||
        (CL > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                       cudaSuccess) ||
        cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess || clusters < 1) {
        cudaGetLastError();
        return false;
    }
    return true;
}

bool dct_loop_configure(int n)
{
#define X(NN, CL) \
    if (n == NN) return dct_loop_configure_t<NN, CL>();
    TVCS_DCT_LOOP_TABLE(X)
#undef X
    return false;
}

cudaError_t launch_dct_loop(int n, const DctLoopArgs& a, cudaStream_t s)
{
#define X(NN, CL)                                                                \
    if (n == NN) {                                                               \
        cudaLaunchAttribute attr;                                                \
        cudaLaunchConfig_t cfg = dct_loop_config<NN, CL>(&attr);                 \
        cfg.stream = s;                                                          \
        return cudaLaunchKernelEx(&cfg, k_dct_loop<NN, CL>, a);                  \
    }
    TVCS_DCT_LOOP_TABLE(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace tvcs
