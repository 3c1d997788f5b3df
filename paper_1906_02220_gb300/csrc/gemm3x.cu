// FP32-accurate GEMM on the tensor cores (sm_103a):
//   C[m][n] = alpha * colscale[n] * sum_k A[m][k] B[k][n]
// for the FP32 contractions of a CTM move in the tensor-core precisions: the
// edge products of the enlarged corners and of the absorption, the subspace
// products M V and M^T U, the basis products, the projectors and the bond metric.
//
// Accuracy.  Every operand is split as x = hi + lo with hi rounded to nearest
// TF32 (|lo| <= 2^-11 |x|), and lo B_hi + hi B_lo + hi B_hi is formed.  The
// tensor core truncates its FP32 accumulator at every instruction, so a sum
// kept there over the whole K loses ~3e-8 of itself per instruction, always
// towards zero.  Here an accumulator holds 32 values of K at most: the small
// products first, then four instructions of hi B_hi, and is then added in FP32
// (rounded to nearest) to the running sum in registers.  Relative
// to FP64 in the Frobenius norm (operands N(0,1), M x N x K): 5184 x 160 x 5184
// 1.9e-7, 9216 x 160 x 9216 2.6e-7, 5184 x 5184 x 144 1.4e-7; FP32 FMAs on the
// CUDA cores 1.3e-6, 1.7e-6, 2.2e-7.  Sums of one sign: 1.5e-7, 1.9e-7, 1.3e-7 against
// 1.1e-6, 1.5e-6, 1.8e-7, from K = 100 down about as the FMAs (64: 1.4e-7, 1.2e-7).
// Where a single product makes up a sum, as in nearly product-like environments,
// an FMA's one rounding is the better (some 2e-8, 4e-8 here).
//
// Time (9216 x 160 x 9216, 27 GFLOP): 111 us, on the CUDA cores 1360 us;
// 5184^3: 1.03 ms = 269 TFLOP/s, 85 % of a third of the TF32 rate, against 1.21 ms
// of a kernel with both split operands in shared memory (whose bandwidth bound it).
//
// Structure.  128 x bn output tiles (bn <= 160), one persistent CTA per SM:
//   warps 0, 2  TMA producers: raw FP32 A tiles (128 x 32) and split B tiles (bn x 32
//               each) into rings of their own: a stage of A is free again once
//               the converters have it in tensor memory, one of B only when its
//               MMAs are done;
//   warp 1      tensor memory; issues the MMAs, A from tensor memory.  All its lanes
//               walk the loop and one issues: with the loop inside a one-lane
//               branch the issue took 1.13 us a K block (12 MMAs) instead of 0.71;
//   warps 4-7   converters: one row of A per thread, split into hi and lo and
//               stored to tensor memory (three buffers).  A never goes back to
//               shared memory, whose bandwidth the MMAs' B reads already fill
//               (bn x 32 bytes per 128 x bn x 8 MMA; with A there too it would be
//               the bound, as in tcgen05.cu);
//   warps 8-15  drain the accumulator (two buffers) into registers after every
//               K block, and store the tile through shared memory.
// A may be row-major ([m][k]) or column-major ([k][m]): the converters read
// either from the staged tile.  B is split and laid out K-major by split_b
// (it is the small operand).  K is split over CTAs when the tiles leave SMs
// idle, with a reduction in a fixed order.  Every wait is bounded; a time-out
// sets bits 64 (producer), 128 (MMA), 256 (converters) or 512 (drain) of *err.
#include <algorithm>
#include <cmath>

#include "tc_ptx.cuh"

#include "engine.cuh"

namespace kh {

// row-major FP32 matrix as a tensor map of 32-column boxes (tcgen05.cu); a
// column-major A is the row-major [K][M] matrix in 32 x 32 boxes
CUtensorMap tc_make_map(const float* p, long long rows, long long K, long long ld, int box_rows);

namespace x3 {

using namespace tc;

constexpr int BM = 128, BK = 32, BNMAX = 160;
constexpr int ASTAGES = 5, BSTAGES = 3, ABUF = 3;
constexpr int A_BYTES = BM * BK * 4, B_BYTES = BNMAX * BK * 4;      // a stage of A; of B hi and of B lo
constexpr int ZROW = 20;                                            // floats per staged output row (16 + 4)
constexpr int Z_BYTES = 8 * 32 * ZROW * 4;
constexpr int SMEM = ASTAGES * A_BYTES + BSTAGES * 2 * B_BYTES + Z_BYTES + 1024;
constexpr int THREADS = 512;
constexpr int C_ACC = 0, C_A = 2 * BNMAX;                           // tensor-memory columns
constexpr int GM = 12;                                              // row tiles walked together (L2 reuse of both operands)

struct Bars {
    uint64_t ra_full[ASTAGES], ra_empty[ASTAGES], b_full[BSTAGES], b_empty[BSTAGES], a_full[ABUF], a_empty[ABUF], acc_full[2], acc_empty[2], drain;
};

struct Work {
    int mt, nt, splits, kb, kper;      // tiles, K splits, K blocks in all and per split
};

// Work item w: K split, then groups of GM row tiles, within a group down the
// rows first.
__device__ __forceinline__ void work_item(const Work& W, int w, int& m, int& n, int& s) {
    const int per = W.mt * W.nt;
    s = w / per;
    w -= s * per;
    const int g = w / (GM * W.nt), m0 = g * GM, gm = min(GM, W.mt - m0);
    w -= g * GM * W.nt;
    m = m0 + w % gm;
    n = w / gm;
}

__device__ __forceinline__ bool wait_all(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

template <bool MMAJOR>
__global__ void __launch_bounds__(THREADS, 1)
gemm3x_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mBh,
              const __grid_constant__ CUtensorMap mBl, float* __restrict__ C, int M, int N, int K, int bn, Work W,
              long long ldc, long long split_stride, float alpha, const float* __restrict__ colscale, int* err) {
    pdl_start();
    extern __shared__ uint8_t smem_raw[];
    __shared__ Bars bars;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = base;
    uint8_t* sB = base + ASTAGES * A_BYTES;
    const int total = W.mt * W.nt * W.splits;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ASTAGES; ++s) {
            mbar_init(&bars.ra_full[s], 1);
            mbar_init(&bars.ra_empty[s], 128);           // the converters
        }
        for (int s = 0; s < BSTAGES; ++s) {
            mbar_init(&bars.b_full[s], 1);
            mbar_init(&bars.b_empty[s], 1);              // the MMAs' completion
        }
        for (int s = 0; s < ABUF; ++s) {
            mbar_init(&bars.a_full[s], 128);
            mbar_init(&bars.a_empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars.acc_full[s], 1);
            mbar_init(&bars.acc_empty[s], 8);            // one arrival per drain warp
        }
        mbar_init(&bars.drain, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;

    if (warp == 0 || warp == 2) {
        // ------------------------------------------------------------ producers (A: warp 0, B: warp 2)
        if (lane == 0) {
            const bool isA = warp == 0;
            const int nst = isA ? ASTAGES : BSTAGES;
            uint64_t* full = isA ? bars.ra_full : bars.b_full;
            uint64_t* empty = isA ? bars.ra_empty : bars.b_empty;
            const uint32_t bytes = isA ? (uint32_t)A_BYTES : 2u * (uint32_t)bn * 128u;
            int s = 0, u = 0, issued = 0;
            bool ok = true;
            for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
                int m, n, sp;
                work_item(W, w, m, n, sp);
                const int kb1 = min(W.kb, (sp + 1) * W.kper);
                for (int kb = sp * W.kper; kb < kb1; ++kb) {
                    if (!mbar_wait(&empty[s], (u & 1) ^ 1, abort_flag)) {
                        s_abort = 1;
                        atomicOr(err, 64);
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(&full[s], bytes);
                    if (!isA) {
                        uint8_t* st = sB + s * 2 * B_BYTES;
                        tma_load_2d(st, &mBh, &full[s], kb * BK, n * bn);
                        tma_load_2d(st + B_BYTES, &mBl, &full[s], kb * BK, n * bn);
                    } else if (MMAJOR) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            tma_load_2d(sA + s * A_BYTES + j * 4096, &mA, &full[s], m * BM + 32 * j, kb * BK);
                    } else {
                        tma_load_2d(sA + s * A_BYTES, &mA, &full[s], kb * BK, m * BM);
                    }
                    ++issued;
                    if (++s == nst) {
                        s = 0;
                        ++u;
                    }
                }
            }
            // copies still in flight land before the CTA exits: the last use of each stage
            for (int q = 0; q < nst && q < issued; ++q) {
                const int last = (issued - 1 - q) / nst;      // number of this stage's last use
                for (uint32_t i = 0; !mbar_try_wait(&full[(issued - 1 - q) % nst], (uint32_t)last & 1); ++i)
                    if (i >= (1u << 22)) {
                        atomicOr(err, 64);
                        break;
                    }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        // the whole warp walks the loop, one lane issues (see elect_one)
        const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(bn >> 3) << 17) |
                               ((uint32_t)(BM >> 4) << 24);
        const uint32_t by = elect_one();
        int it = 0, s = 0, su = 0, a = 0, au = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            int m, n, sp;
            work_item(W, w, m, n, sp);
            const int kb1 = min(W.kb, (sp + 1) * W.kper);
            for (int kb = sp * W.kper; kb < kb1; ++kb, ++it) {
                const int c = it & 1;
                if (!wait_all(&bars.b_full[s], su & 1, abort_flag) || !wait_all(&bars.a_full[a], au & 1, abort_flag) ||
                    !wait_all(&bars.acc_empty[c], ((it >> 1) & 1) ^ 1, abort_flag)) {
                    s_abort = 1;
                    if (lane == 0) atomicOr(err, 128);
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t d = tmem + C_ACC + c * BNMAX;
                const uint32_t ah = tmem + C_A + a * 2 * BK, al = ah + BK;
                const uint64_t bh = smem_desc(smem_u32(sB + s * 2 * B_BYTES));
                const uint64_t bl = smem_desc(smem_u32(sB + s * 2 * B_BYTES + B_BYTES));
                // the small products first: the truncated accumulator is then still
                // small.  A K step is 8 columns of A and 32 bytes (2 descriptor units) of B.
                if (K - kb * BK >= BK) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_tf32_tmem_a(by, d, al + ks * 8, bh + ks * 2, idesc, ks > 0 ? 1u : 0u);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) umma_tf32_tmem_a(by, d, ah + ks * 8, bl + ks * 2, idesc, 1u);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) umma_tf32_tmem_a(by, d, ah + ks * 8, bh + ks * 2, idesc, 1u);
                } else {
                    const int steps = (K - kb * BK + 7) / 8;
                    for (int ks = 0; ks < steps; ++ks)
                        umma_tf32_tmem_a(by, d, al + ks * 8, bh + ks * 2, idesc, ks > 0 ? 1u : 0u);
                    for (int ks = 0; ks < steps; ++ks) umma_tf32_tmem_a(by, d, ah + ks * 8, bl + ks * 2, idesc, 1u);
                    for (int ks = 0; ks < steps; ++ks) umma_tf32_tmem_a(by, d, ah + ks * 8, bh + ks * 2, idesc, 1u);
                }
                umma_commit(by, &bars.a_empty[a]);
                umma_commit(by, &bars.b_empty[s]);
                umma_commit(by, &bars.acc_full[c]);
                if (++s == BSTAGES) {
                    s = 0;
                    ++su;
                }
                if (++a == ABUF) {
                    a = 0;
                    ++au;
                }
            }
        }
        // every MMA issued completes before tensor memory is freed
        umma_commit(by, &bars.drain);
        for (uint32_t i = 0; !mbar_try_wait(&bars.drain, 0); ++i)
            if (i >= (1u << 22)) {
                if (lane == 0) atomicOr(err, 128);
                break;
            }
    } else if (warp >= 4 && warp < 8) {
        // ------------------------------------------------------------ converters
        const int q = warp & 3, t = 32 * q + lane;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        int it = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            int m, n, sp;
            work_item(W, w, m, n, sp);
            const int kb1 = min(W.kb, (sp + 1) * W.kper);
            for (int kb = sp * W.kper; kb < kb1; ++kb, ++it) {
                const int s = it % ASTAGES, a = it % ABUF;
                if (!wait_all(&bars.ra_full[s], (it / ASTAGES) & 1, abort_flag)) { ok = false; break; }
                const uint8_t* st = sA + s * A_BYTES;
                float x[BK];
                if (MMAJOR) {
                    // 32 x 32 boxes [k][m]: lanes along m
                    const uint8_t* b = st + q * 4096 + (lane & 3) * 4;
#pragma unroll
                    for (int k = 0; k < BK; ++k)
                        x[k] = *(const float*)(b + k * 128 + ((((uint32_t)lane >> 2) ^ (k & 7)) << 4));
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 v = *(const float4*)(st + t * 128 + ((j ^ (t & 7)) << 4));
                        x[4 * j] = v.x;
                        x[4 * j + 1] = v.y;
                        x[4 * j + 2] = v.z;
                        x[4 * j + 3] = v.w;
                    }
                }
                float big = 0.f;
#pragma unroll
                for (int k = 0; k < BK; ++k) big = fmaxf(big, fabsf(x[k]));
                const uint32_t half = tf32_half(big);
                if (!wait_all(&bars.a_empty[a], ((it / ABUF) & 1) ^ 1, abort_flag)) { ok = false; break; }
                fence_after();
                const uint32_t dst = tmem + lane_base + C_A + a * 2 * BK;
#pragma unroll
                for (int c0 = 0; c0 < BK; c0 += 16) {
                    float hi[16], lo[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        hi[i] = tf32_head(x[c0 + i], half);
                        lo[i] = x[c0 + i] - hi[i];
                    }
                    tmem_st16(dst + c0, hi);
                    tmem_st16(dst + BK + c0, lo);
                }
                tmem_st_wait();
                fence_before();
                mbar_arrive(&bars.a_full[a]);
                // only now have the loads of x provably completed: with the arrival right
                // after them, and the wait on a_empty behind it, pieces of the stage's next
                // tile were read instead (while the drain stored a tile)
                mbar_arrive(&bars.ra_empty[s]);
            }
        }
        if (!ok) {
            s_abort = 1;
            if (lane == 0) atomicOr(err, 256);
        }
    } else if (warp >= 8) {
        // ------------------------------------------------------------ drain and store
        const int q = warp & 3, dg = (warp - 8) >> 2;      // tensor-memory quadrant, column group parity
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        float* zs = (float*)(sB + BSTAGES * 2 * B_BYTES) + (warp - 8) * 32 * ZROW;
        constexpr int NJ = BNMAX / 32;                     // 16-column groups of this warp
        const int ng = bn / 16;
        int it = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            int m, n, sp;
            work_item(W, w, m, n, sp);
            const int kb0 = sp * W.kper, kb1 = min(W.kb, kb0 + W.kper);
            float acc[NJ][16];
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[j][i] = 0.f;
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                const int c = it & 1;
                if (!wait_all(&bars.acc_full[c], (it >> 1) & 1, abort_flag)) { ok = false; break; }
                fence_after();
                // two column groups in flight: the register file holds acc and 32 more
                constexpr int NB = (NJ + 1) / 2;
#pragma unroll
                for (int jb = 0; jb < NB; ++jb) {
                    uint32_t r[2][16];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int j = 2 * jb + e;
                        if (j < NJ && 2 * j + dg < ng)
                            tmem_ld16_async(tmem + lane_base + C_ACC + c * BNMAX + (2 * j + dg) * 16, r[e]);
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int j = 2 * jb + e;
                        if (j < NJ && 2 * j + dg < ng) {
                            tmem_regs_ready(r[e]);
#pragma unroll
                            for (int i = 0; i < 16; ++i) acc[j < NJ ? j : 0][i] += __uint_as_float(r[e][i]);
                        }
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.acc_empty[c]);
            }
            if (!ok) break;
            float* Cs = C + sp * split_stride;
            const int row0 = m * BM + 32 * q;
            const bool vec = (ldc & 3) == 0 && ((uintptr_t)Cs & 15) == 0;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                if (2 * j + dg >= ng) continue;
                const int col0 = n * bn + (2 * j + dg) * 16;
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *(float4*)(zs + lane * ZROW + i) = make_float4(acc[j][i], acc[j][i + 1], acc[j][i + 2], acc[j][i + 3]);
                __syncwarp();
                if (vec && col0 + 16 <= N) {
                    const int cc = col0 + 4 * (lane & 3);
                    float4 sc = make_float4(alpha, alpha, alpha, alpha);
                    if (colscale)
                        sc = make_float4(alpha * colscale[cc], alpha * colscale[cc + 1], alpha * colscale[cc + 2],
                                         alpha * colscale[cc + 3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rr = 8 * i + (lane >> 2);
                        float4 v = *(const float4*)(zs + rr * ZROW + 4 * (lane & 3));
                        v = make_float4(v.x * sc.x, v.y * sc.y, v.z * sc.z, v.w * sc.w);
                        if (row0 + rr < M) *(float4*)(Cs + (long long)(row0 + rr) * ldc + cc) = v;
                    }
                } else {
                    const int cc = col0 + (lane & 15);
                    const float sc = cc < N ? (colscale ? alpha * colscale[cc] : alpha) : 0.f;
                    for (int i = 0; i < 16; ++i) {
                        const int rr = 2 * i + (lane >> 4);
                        if (row0 + rr < M && cc < N)
                            Cs[(long long)(row0 + rr) * ldc + cc] = sc * zs[rr * ZROW + (lane & 15)];
                    }
                }
            }
        }
        if (!ok) {
            s_abort = 1;
            if (lane == 0) atomicOr(err, 512);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// B (N x K by strides) into its K-major hi and lo parts (row stride ld >= K,
// a multiple of 4; the columns past K are not written, nor read: the tensor maps
// are K wide, and where the last step of eight values runs past K the copies
// fill in zeros).  32 x 32 tiles through shared memory, so that both sides are
// coalesced.
__global__ void __launch_bounds__(256)
split_b_kernel(const float* __restrict__ B, long long sn, long long sk, int N, int K, float* __restrict__ hi,
               float* __restrict__ lo, int ld) {
    pdl_start();
    __shared__ float t[32][33];
    const int n0 = blockIdx.y * 32, k0 = blockIdx.x * 32;
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    for (int i = ly; i < 32; i += 8) {
        const int n = n0 + (sn == 1 ? lx : i), k = k0 + (sn == 1 ? i : lx);
        const float v = (n < N && k < K) ? B[n * sn + k * sk] : 0.f;
        t[sn == 1 ? lx : i][sn == 1 ? i : lx] = v;
    }
    __syncthreads();
    for (int i = ly; i < 32; i += 8) {
        const int n = n0 + i, k = k0 + lx;
        if (n < N && k < K) {
            const float v = t[i][lx], h = tf32_head(v, tf32_half(fabsf(v)));
            hi[(long long)n * ld + k] = h;
            lo[(long long)n * ld + k] = v - h;
        }
    }
}

__global__ void reduce_kernel(const float* __restrict__ part, int splits, long long stride, int M, int N, int ldp,
                              float* __restrict__ C, long long ldc, float alpha, const float* __restrict__ colscale) {
    pdl_start();
    const long long tot = (long long)M * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
        const int m = (int)(i / N), n = (int)(i % N);
        const float* p = part + (long long)m * ldp + n;
        float a = 0.f;
        for (int s = 0; s < splits; ++s) a += p[s * stride];
        C[m * ldc + n] = (colscale ? alpha * colscale[n] : alpha) * a;
    }
}

// Tile width, K splits and the estimated time (us): a tile's K block takes the
// MMAs' time (12 of 128 x bn x 8, half a clock per column) or, for narrow tiles,
// the converters' and the drain's latency (~0.3 us); a work item ~1.5 us of
// pipeline fill and stores; a split adds the partial sums' round trip.
struct Plan {
    int bn;
    Work W;
    double us;
};
Plan make_plan(int M, int N, int K, long long sk_elems, int sms) {
    Plan best{};
    best.us = 1e30;
    const int mt = (M + BM - 1) / BM, kb = (K + BK - 1) / BK;
    const int n16 = (N + 15) / 16 * 16;
    for (int bn = std::min(BNMAX, n16); bn >= std::min(96, n16); bn -= 16) {
        const int nt = (N + bn - 1) / bn;
        for (int s = 1; s <= 16 && s <= kb; ++s) {
            const int kper = (kb + s - 1) / s, sp = (kb + kper - 1) / kper;
            if (sp != s) continue;
            const long long ldp = (N + 3) / 4 * 4;
            if (s > 1 && (long long)s * M * ldp > sk_elems) continue;
            const double waves = std::ceil((double)mt * nt * s / sms);
            const double block = std::max(0.3, 12.0 * bn / 2 / 1900.0);
            double us = waves * (kper * block + 1.5);
            if (s > 1) us += 3.0 + (double)s * M * N * 8.0 / 6e6;
            if (us < best.us) best = Plan{bn, Work{mt, nt, s, kb, kper}, us};
        }
    }
    return best;
}

}  // namespace x3

void gemm3x_split_b(const float* B, long long sn, long long sk, int N, int K, float* hi, float* lo, int ld,
                    cudaStream_t st) {
    dim3 grid((K + 31) / 32, (N + 31) / 32);
    launch(x3::split_b_kernel, grid, 256, 0, st, B, sn, sk, N, K, hi, lo, ld);
}

bool gemm3x_usable(const float* A, long long lda) { return ((uintptr_t)A & 15) == 0 && lda % 4 == 0; }

void gemm3x(const float* A, long long lda, bool a_mmajor, const float* Bhi, const float* Blo, int ldb, float* C,
            int M, int N, int K, long long ldc, float alpha, const float* colscale, float* sk, long long sk_elems,
            int* err, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return;
    const int sms = device_sms();
    const x3::Plan p = x3::make_plan(M, N, K, sk ? sk_elems : 0, sms);
    const CUtensorMap ma = a_mmajor ? tc_make_map(A, K, M, lda, 32) : tc_make_map(A, M, K, lda, x3::BM);
    const CUtensorMap mh = tc_make_map(Bhi, N, K, ldb, p.bn), ml = tc_make_map(Blo, N, K, ldb, p.bn);
    const int total = p.W.mt * p.W.nt * p.W.splits, grid = std::min(total, sms);
    const bool split = p.W.splits > 1;
    const int ldp = (N + 3) / 4 * 4;
    float* out = split ? sk : C;
    const long long ldo = split ? ldp : ldc, stride = split ? (long long)M * ldp : 0;
    const float al = split ? 1.f : alpha;
    const float* cs = split ? nullptr : colscale;
    static std::atomic<size_t> granted[2][kMaxDevices] = {};
    if (a_mmajor) {
        smem_opt_in(x3::gemm3x_kernel<true>, (size_t)x3::SMEM, granted[1]);
        launch(x3::gemm3x_kernel<true>, grid, x3::THREADS, x3::SMEM, st, ma, mh, ml, out, M, N, K, p.bn, p.W, ldo, stride,
                                                                     al, cs, err);
    } else {
        smem_opt_in(x3::gemm3x_kernel<false>, (size_t)x3::SMEM, granted[0]);
        launch(x3::gemm3x_kernel<false>, grid, x3::THREADS, x3::SMEM, st, ma, mh, ml, out, M, N, K, p.bn, p.W, ldo,
                                                                      stride, al, cs, err);
    }
    if (split) {
        launch(x3::reduce_kernel, grid_for((long long)M * N), 256, 0, st, sk, p.W.splits, stride, M, N, ldp, C, ldc, alpha,
                                                                      colscale);
    }
}

}  // namespace kh
