// Layered (ket layer, then bra layer) site contraction of the enlarged
// corners and edge absorptions, Fig. 4 and Sec. III of arXiv:1906.02220, as
// one persistent tcgen05 kernel for sm_103a.  The shapes, the operand images
// and the index conventions are in layered.cuh.
//
// One CTA per SM loops over tiles of 128 rows (b, ib) (bt = 128 / D^2 blocks
// b per tile).  Per tile and chunk c of pc physical indices:
//   warp 0 (lanes 0, 1)  bulk-copies the chunk's ket (B1) and bra (B2) operand
//                        images into shared-memory rings (or once, when all
//                        chunks fit: resident images);
//   warp 1               tensor memory; issues the ket GEMMs
//                          acc1[c % nb1] = Y_tile * B1_c
//   warp 2               issues the bra GEMMs
//                          out         += Z_c   * B2_c
//                        (both with A in tensor memory, one elected lane issuing,
//                        each group committed to an mbarrier);
//   warps 4-7, 8-11      two worker sets, taking chunks in turn: read acc1 row
//                        (b, ib) per thread, scatter it into a shared-memory
//                        buffer in (b, ok) row order, read back row (b, ok), split
//                        it into TF32 hi/lo (or round it to BF16 pairs) and store it
//                        to tensor memory as the bra GEMM's A operand.  The first
//                        set also loads the next Y tile into tensor memory (one row
//                        per thread) and stores the output rows.
// With 3 passes every product is A_hi B_hi + A_hi B_lo + A_lo B_hi from operands
// rounded to nearest TF32; the ket accumulator takes the two small ones first, the
// bra GEMM has an accumulator for them (the tensor core truncates the accumulator
// at every instruction).  Up to D = 5 the order is the fixed one (layered.cuh).  BF16 runs one kind::f16 pass (K = 16 per MMA).
// What bounds it: the tensor pipe's narrow MMAs at D >= 6 (73 % of the TF32 rate
// over the padded shapes at D = 8), the chunk's chain of hand-offs below.  Time of a
// launch, 3xTF32, p = 16: (4, 64) 21.5 us, (5, 100) 134, (6, 144) 443 (140 TFLOP/s),
// (8, 144) 1481 (235); with Y as a shared-memory operand, one worker set and MMAs
// issued from a one-lane branch: 25.5, 167, 722, 2113.  Y in tensor memory frees
// 64 KB for two stages of both image rings, whose reload was on the chain.
// Every wait is bounded: on time-out the kernel raises a flag, the roles drain,
// tensor memory is freed and the kernel
// returns with bits set in *err (8 producer, 16 MMA issuer, 32 workers).
#include <atomic>
#include <type_traits>

#include <cuda_bf16.h>

#include "engine.cuh"
#include "layered.cuh"
#include "tc_ptx.cuh"

namespace kh {

namespace lay {

using namespace tc;

constexpr int NSET = 2;                         // worker sets (4 warps each)
constexpr int WORKER0 = 4;                      // first worker warp (its tensor-memory quadrant is its number mod 4)
constexpr int THREADS = 32 * WORKER0 + 128 * NSET;
constexpr int MAXST = 16;

// instruction descriptor: FP32 accumulator, A and B TF32 (kind::tf32) or BF16
// (kind::f16), K-major, N and M = 128
constexpr uint32_t idesc(int n, bool bf16) {
    const uint32_t fmt = bf16 ? 1u : 2u;
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// packs two FP32 values as BF16 (round to nearest even), a in the low half
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(a));
    const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(b));
    return lo | (hi << 16);
}

struct Bars {
    uint64_t b1_full[MAXST], b1_empty[MAXST], b2_full[MAXST], b2_empty[MAXST];
    uint64_t acc1_full[2], acc1_empty[2], a2_full[2], a2_empty[2];
    uint64_t zs_w[NSET], zs_r[NSET];
    uint64_t y_full, y_empty, out_full, out_empty, drain[2];
};

// Bounded wait made uniform over the warp: false on time-out or abort.
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
    const bool ok = mbar_wait(bar, parity, abort_flag);
    return __all_sync(0xffffffffu, ok);
}

// Wait that ignores the abort flag (used while draining).
__device__ __forceinline__ bool wait_drain(uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < (1u << 22); ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

template <int D, int NPASS, bool BF>
__global__ void __launch_bounds__(THREADS, 1)
layered_kernel(const float* __restrict__ Y, long long nb, int nc, const uint8_t* __restrict__ img1,
               const uint8_t* __restrict__ img2, float* __restrict__ out, int ntiles, int nst1, int nst2,
               int* err) {
    pdl_start();
    static_assert(!BF || NPASS == 1, "BF16 runs one pass");
    constexpr Plan P = make_plan(D, NPASS, BF);
    constexpr int D2 = P.d2;
    constexpr int NPL = NPASS == 3 ? 2 : 1;
    constexpr int KS = P.kstep;
    constexpr uint32_t ID1 = idesc(P.n1p, BF), ID2 = idesc(P.n2p, BF);
    constexpr int B1_SZ = NPL * P.b1_bytes, B2_SZ = NPL * P.b2_bytes;

    extern __shared__ uint8_t smem_raw[];
    __shared__ Bars bars;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool res1 = nst1 == nc, res2 = nst2 == nc;      // images loaded once
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sB1 = base;
    uint8_t* sB2 = sB1 + (size_t)nst1 * B1_SZ;
    float* sZ = (float*)(sB2 + (size_t)nst2 * B2_SZ);

    if (threadIdx.x == 0) {
        for (int s = 0; s < MAXST; ++s) {
            mbar_init(&bars.b1_full[s], 1);
            mbar_init(&bars.b1_empty[s], 1);
            mbar_init(&bars.b2_full[s], 1);
            mbar_init(&bars.b2_empty[s], 1);
        }
        for (int j = 0; j < 2; ++j) {
            mbar_init(&bars.acc1_full[j], 1);
            mbar_init(&bars.acc1_empty[j], 128);
            mbar_init(&bars.a2_full[j], 128);
            mbar_init(&bars.a2_empty[j], 1);
        }
        mbar_init(&bars.y_full, 128);
        mbar_init(&bars.y_empty, 1);
        mbar_init(&bars.out_full, 1);
        mbar_init(&bars.out_empty, 128);
        for (int s = 0; s < NSET; ++s) {
            mbar_init(&bars.zs_w[s], 128);
            mbar_init(&bars.zs_r[s], 128);
        }
        for (int q = 0; q < 2; ++q) mbar_init(&bars.drain[q], 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"((uint32_t)P.tmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* abort_flag = &s_abort;

    if (warp == 0) {
        // ---------------------------------------------------------- producer
        if (lane < 2) {
            const bool ket = lane == 0;
            const int nst = ket ? nst1 : nst2;
            const bool res = ket ? res1 : res2;
            const int sz = ket ? B1_SZ : B2_SZ;
            uint8_t* ring = ket ? sB1 : sB2;
            const uint8_t* img = ket ? img1 : img2;
            uint64_t* full = ket ? bars.b1_full : bars.b2_full;
            uint64_t* empty = ket ? bars.b1_empty : bars.b2_empty;
            int armed[MAXST];
            for (int s = 0; s < MAXST; ++s) armed[s] = 0;
            if (res) {
                if (blockIdx.x < ntiles)
                    for (int c = 0; c < nc; ++c) {
                        mbar_expect_tx(&full[c], (uint32_t)sz);
                        bulk_load(ring + (size_t)c * sz, img + (size_t)c * sz, (uint32_t)sz, &full[c]);
                        armed[c] = 1;
                    }
            } else {
                long long g = 0;
                for (int tile = blockIdx.x; tile < ntiles && !*abort_flag; tile += gridDim.x) {
                    for (int c = 0; c < nc; ++c, ++g) {
                        const int s = (int)(g % nst);
                        const uint32_t u = (uint32_t)(g / nst);
                        if (!mbar_wait(&empty[s], (u & 1) ^ 1, abort_flag)) {
                            s_abort = 1;
                            atomicOr(err, 8);
                            break;
                        }
                        mbar_expect_tx(&full[s], (uint32_t)sz);
                        bulk_load(ring + (size_t)s * sz, img + (size_t)c * sz, (uint32_t)sz, &full[s]);
                        armed[s] = (int)u + 1;
                    }
                }
            }
            // copies still in flight land before the CTA exits
            for (int s = 0; s < MAXST; ++s)
                if (armed[s] && !wait_drain(&full[s], (uint32_t)(armed[s] - 1) & 1)) atomicOr(err, 8);
        }
    } else if (warp <= 2) {
        // ---------------------------------------------------------- MMA issuers
        // A warp walks its loop whole and one lane issues: in a one-lane branch
        // every MMA's operands are moved to uniform registers first, ~50 ns an
        // MMA, which is longer than these narrow MMAs take.
        bool ok = true;
        long long g0 = 0;
        int it = 0;
        const uint32_t by = elect_one();
        constexpr int S1 = P.k1p / KS, S2 = P.k2p / KS;       // K steps of the two GEMMs
        if (warp == 1) {
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it, g0 += nc) {
                if (!wait_warp(&bars.y_full, it & 1, abort_flag)) { ok = false; break; }
                fence_after();
                for (int c = 0; c < nc; ++c) {                      // ket layer of chunk c
                    const long long g = g0 + c;
                    const int s1 = res1 ? c : (int)(g % nst1);
                    const uint32_t ph1 = res1 ? 0u : (uint32_t)((g / nst1) & 1);
                    const int j = (int)(g % P.nb1);
                    const long long h = g - P.nb1;              // the chunk that had this accumulator
                    if (!wait_warp(&bars.b1_full[s1], ph1, abort_flag) ||
                        (h >= 0 && !wait_warp(&bars.acc1_empty[h & 1], (uint32_t)((h >> 1) & 1), abort_flag))) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint32_t d0 = tmem + P.c_acc1 + j * P.nacc1 * P.acc1_cols, y = tmem + P.c_y;
                    const uint64_t db0 = smem_desc(smem_u32(sB1 + (size_t)s1 * B1_SZ));
                    // lo B_hi, hi B_lo, hi B_hi with 3 passes (the reverse in the fixed
                    // order), hi B_hi alone with one
#pragma unroll
                    for (int pq = 0; pq < NPASS; ++pq) {
                        const int pass = P.fixed ? 2 - pq : 3 - NPASS + pq;
#pragma unroll
                        for (int ks = 0; ks < S1; ++ks) {
                            const int i = pq * S1 + ks;
                            const uint32_t d = d0 + (i % P.nacc1) * P.acc1_cols;
                            // 32 bytes of K per MMA, four per 128-byte block (16-byte descriptor units)
                            const uint64_t db = db0 + ((pass == 1 ? P.b1_bytes : 0) + (ks >> 2) * (P.n1p * 128) + (ks & 3) * 32) / 16;
                            const uint32_t a = y + (NPASS == 3 && pass == 0 ? P.y_cols : 0) + ks * 8;
                            const uint32_t acc = i >= P.nacc1 ? 1u : 0u;
                            if constexpr (BF) umma_f16_tmem_a(by, d, a, db, ID1, acc);
                            else umma_tf32_tmem_a(by, d, a, db, ID1, acc);
                        }
                    }
                    umma_commit(by, &bars.acc1_full[g & 1]);
                    if (!res1) umma_commit(by, &bars.b1_empty[s1]);
                    if (c == nc - 1) umma_commit(by, &bars.y_empty);
                }
            }
        } else {
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it, g0 += nc) {
                for (int cc = 0; cc < nc; ++cc) {                   // bra layer of chunk cc
                    const long long g = g0 + cc;
                    const int s2 = res2 ? cc : (int)(g % nst2);
                    const uint32_t ph2 = res2 ? 0u : (uint32_t)((g / nst2) & 1);
                    const int ja = (int)(g % P.na2);
                    const uint32_t pa = (uint32_t)((g / P.na2) & 1);
                    if (!wait_warp(&bars.b2_full[s2], ph2, abort_flag) || !wait_warp(&bars.a2_full[ja], pa, abort_flag) ||
                        (cc == 0 && !wait_warp(&bars.out_empty, (uint32_t)(it & 1) ^ 1, abort_flag))) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint32_t d0 = tmem + P.c_out;
                    const uint32_t a2 = tmem + P.c_a2 + ja * NPL * P.a2_cols;
                    const uint64_t db0 = smem_desc(smem_u32(sB2 + (size_t)s2 * B2_SZ));
#pragma unroll
                    for (int pq = 0; pq < NPASS; ++pq) {
                        const int pass = P.fixed ? 2 - pq : 3 - NPASS + pq;
#pragma unroll
                        for (int ks = 0; ks < S2; ++ks) {
                            const int i = pq * S2 + ks;
                            const uint64_t db = db0 + ((pass == 1 ? P.b2_bytes : 0) + (ks >> 2) * (P.n2p * 128) + (ks & 3) * 32) / 16;
                            // 8 tensor-memory columns of Z per MMA (8 TF32 or 16 BF16 values)
                            const uint32_t a = a2 + (NPASS == 3 && pass == 0 ? P.a2_cols : 0) + ks * 8;
                            const bool main = pass == 2;            // leading products: accumulators 0 .. nm - 1
                            const uint32_t dd = d0 + (P.fixed ? i % P.nacc2 : main ? ks % P.nm : P.nm) * P.out_cols;
                            const bool first = P.fixed ? i < P.nacc2 : main ? ks < P.nm : (pass == 0 && ks == 0);
                            const uint32_t acc = (cc > 0 || !first) ? 1u : 0u;
                            if constexpr (BF) umma_f16_tmem_a(by, dd, a, db, ID2, acc);
                            else umma_tf32_tmem_a(by, dd, a, db, ID2, acc);
                        }
                    }
                    umma_commit(by, &bars.a2_empty[g & 1]);
                    if (!res2) umma_commit(by, &bars.b2_empty[s2]);
                    if (cc == nc - 1) umma_commit(by, &bars.out_full);
                }
            }
        }
        if (!ok) {
            s_abort = 1;
            if (lane == 0) atomicOr(err, 16);
        }
        // every MMA this warp issued completes before tensor memory is freed
        uint64_t* dr = &bars.drain[warp - 1];
        umma_commit(by, dr);
        if (!wait_drain(dr, 0) && lane == 0) atomicOr(err, 16);
    } else if (warp >= WORKER0) {
        // ---------------------------------------------------------- workers
        const int set = (warp - WORKER0) >> 2;           // chunks g with g % NSET == set
        const int q = warp & 3;                          // tensor-memory lane quadrant
        const int t = 32 * q + lane;                     // tile row of this thread
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const long long total_rows = nb * D2;
        float* zbuf = sZ + set * 128 * P.zs;
        bool ok = true;

        // n values v(i) as A operand columns: TF32 hi columns at `dst`, lo columns
        // npad columns on with 3 passes; or BF16 pairs, the lower index in the low half
        auto store_a = [&](uint32_t dst, auto npad_c, int lo_off, const float* v) {
            constexpr int NP = decltype(npad_c)::value;   // columns (a multiple of 8)
            uint32_t half = 0;                            // heads to nearest, or in the fixed order the leading bits
            if constexpr (NPASS == 3 && D > kFixedOrderD) {
                float big = 0.f;
#pragma unroll
                for (int i = 0; i < NP; ++i) big = fmaxf(big, fabsf(v[i]));
                half = tf32_half(big);
            }
            auto col = [&](int c, bool lo) {
                if constexpr (BF) return __uint_as_float(pack_bf16x2(v[2 * c], v[2 * c + 1]));
                const float x = v[c];
                if (NPASS != 3) return x;
                const float h = tf32_head(x, half);
                return lo ? x - h : h;
            };
#pragma unroll
            for (int l = 0; l < NPL; ++l) {
#pragma unroll
                for (int c0 = 0; c0 + 16 <= NP; c0 += 16) {
                    float w[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) w[i] = col(c0 + i, l == 1);
                    tmem_st16(dst + l * lo_off + c0, w);
                }
                if constexpr (NP % 16 != 0) {
                    float w[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) w[i] = col(NP - 8 + i, l == 1);
                    tmem_st8(dst + l * lo_off + NP - 8, w);
                }
            }
        };
        // one row of the tile's Y into tensor memory (zero past the rows)
        auto load_y = [&](int tile) {
            constexpr int NV = P.k1p;
            float y[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) y[i] = 0.f;
            const long long row = (long long)tile * P.rows + t;
            if (t < P.rows && row < total_rows) {
                const float* src = Y + row * D2;
                if constexpr (D2 % 4 == 0) {
#pragma unroll
                    for (int i = 0; i < D2; i += 4) {
                        const float4 w = __ldg((const float4*)(src + i));
                        y[i] = w.x;
                        y[i + 1] = w.y;
                        y[i + 2] = w.z;
                        y[i + 3] = w.w;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < D2; ++i) y[i] = __ldg(src + i);
                }
            }
            store_a(tmem + lane_base + P.c_y, std::integral_constant<int, P.y_cols>{}, P.y_cols, y);
            tmem_st_wait();
            fence_before();
            mbar_arrive(&bars.y_full);
        };

        if (set == 0 && (int)blockIdx.x < ntiles) load_y(blockIdx.x);
        long long g0 = 0;
        int it = 0;
        uint32_t zcount = 0;                             // chunks this set has transposed
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++it, g0 += nc) {
            const int next = tile + gridDim.x;
            // set 0 loads the next tile's Y (asked into L2 now) and stores this
            // tile's output.  One set does it for every tile: it then waits for
            // every phase of y_empty and out_full, while a wait by parity that
            // skips a phase could return on the one before.
            if (set == 0 && next < ntiles) {
                const long long row = (long long)next * P.rows + t;
                if (t < P.rows && row < total_rows) {
                    const float* src = Y + row * D2;
#pragma unroll
                    for (int i = 0; i < D2; i += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + i));
                }
            }
            for (int c = 0; c < nc && ok; ++c) {
                const long long g = g0 + c;
                if ((int)(g % NSET) != set) continue;
                // ---- ket accumulator row (b, ib) -> transpose buffer rows (b, ok)
                // (chunks signal two barriers in turn, one for each set, whatever the
                // number of buffers: a set then waits for every phase of its own)
                const int j = (int)(g % P.nb1);
                if (!wait_warp(&bars.acc1_full[g & 1], (uint32_t)((g >> 1) & 1), abort_flag)) { ok = false; break; }
                fence_after();
                uint32_t vr[P.n1p / 16][16];
#pragma unroll
                for (int c0 = 0; c0 < P.n1p; c0 += 16)
                    tmem_ld16_async(tmem + lane_base + (uint32_t)(P.c_acc1 + j * P.nacc1 * P.acc1_cols + c0), vr[c0 / 16]);
                tmem_ld_wait();
#pragma unroll
                for (int c0 = 0; c0 < P.n1p; c0 += 16) tmem_regs_ready(vr[c0 / 16]);
                if constexpr (P.nacc1 == 2) {            // 16 columns at a time: the register file
#pragma unroll
                    for (int c0 = 0; c0 < P.n1p; c0 += 16) {
                        uint32_t r[16];
                        tmem_ld16_async(tmem + lane_base + (uint32_t)(P.c_acc1 + (j * 2 + 1) * P.acc1_cols + c0), r);
                        tmem_ld_wait();
                        tmem_regs_ready(r);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            vr[c0 / 16][i] = __float_as_uint(__uint_as_float(vr[c0 / 16][i]) + __uint_as_float(r[i]));
                    }
                }
                auto v = [&](int n) { return __uint_as_float(vr[n >> 4][n & 15]); };
                fence_before();
                mbar_arrive(&bars.acc1_empty[g & 1]);
                // the set's previous chunk has been read out of the buffer
                if (zcount > 0 && !wait_warp(&bars.zs_r[set], (zcount - 1) & 1, abort_flag)) { ok = false; break; }
                if (t < P.rows) {
                    const int b = t / D2, ib = t % D2;
                    float* zrow = zbuf + b * D2 * P.zs;
                    constexpr int NCH = P.pc >= 4 ? P.pc / 4 : 1;   // 16-byte chunks this row's values span
                    // chunk of the values, with the permutation by row & 7 = (b D^2 & 7) ^ ok
                    // (D^2 is 4 or a multiple of 8 where the chunks are permuted)
                    const int ch0 = ((ib * P.pc) >> 2) ^ (P.zswz ? (b * D2) & 7 : 0);
                    int xo[P.zswz ? 8 : 1];
                    if constexpr (P.zswz && NCH == 1) {
#pragma unroll
                        for (int m = 0; m < 8; ++m) xo[m] = ((ch0 ^ m) << 2) + ((ib * P.pc) & 3);
                    }
#pragma unroll
                    for (int ok_ = 0; ok_ < D2; ++ok_) {
#pragma unroll
                        for (int e = 0; e < NCH; ++e) {
                            float* dst;
                            if constexpr (P.zswz && NCH == 1) dst = zrow + ok_ * P.zs + xo[ok_ & 7];
                            else if constexpr (P.zswz) dst = zrow + ok_ * P.zs + ((ch0 ^ e ^ (ok_ & 7)) << 2);
                            else dst = zrow + ok_ * P.zs + ib * P.pc + 4 * e;
                            if constexpr (P.pc >= 4)
                                *(float4*)dst = make_float4(v(4 * e * D2 + ok_), v((4 * e + 1) * D2 + ok_),
                                                            v((4 * e + 2) * D2 + ok_), v((4 * e + 3) * D2 + ok_));
                            else if constexpr (P.pc == 2) *(float2*)dst = make_float2(v(ok_), v(D2 + ok_));
                            else *dst = v(ok_);
                        }
                    }
                }
                mbar_arrive(&bars.zs_w[set]);
                if (!wait_warp(&bars.zs_w[set], zcount & 1, abort_flag)) { ok = false; break; }
                // ---- row (b, ok) of Z -> tensor memory (bra GEMM A operand)
                constexpr int K2R = pad_to(P.k2, 4);          // values read per row
                float z[P.k2p];
#pragma unroll
                for (int i = 0; i < P.k2p; ++i) z[i] = 0.f;
                if (t < P.rows) {
                    const float* src = zbuf + t * P.zs;
                    int xo[8];
#pragma unroll
                    for (int m = 0; m < 8; ++m) xo[m] = (P.zswz ? m ^ (t & 7) : m) << 2;
#pragma unroll
                    for (int i = 0; i < K2R; i += 4) {
                        const float4 w = *(const float4*)(src + (i & ~31) + xo[(i >> 2) & 7]);
                        z[i] = w.x;
                        if (i + 1 < P.k2) z[i + 1] = w.y;
                        if (i + 2 < P.k2) z[i + 2] = w.z;
                        if (i + 3 < P.k2) z[i + 3] = w.w;
                    }
                }
                // the bra GEMM of chunk g - na2 has read this Z buffer
                const int ja = (int)(g % P.na2);
                const long long h = g - P.na2;
                if (h >= 0 && !wait_warp(&bars.a2_empty[h & 1], (uint32_t)((h >> 1) & 1), abort_flag)) {
                    ok = false;
                    break;
                }
                fence_after();
                store_a(tmem + lane_base + (uint32_t)(P.c_a2 + ja * NPL * P.a2_cols),
                        std::integral_constant<int, P.a2_cols>{}, P.a2_cols, z);
                tmem_st_wait();
                fence_before();
                mbar_arrive(&bars.a2_full[ja]);
                // the reads of zbuf have provably completed only now that z is in tensor
                // memory; other warps of the set scatter their next chunk over it then
                mbar_arrive(&bars.zs_r[set]);
                ++zcount;
            }
            if (!ok) break;
            if (set != 0) continue;
            // ---- next tile's Y once the ket GEMMs of this tile have read it
            if (next < ntiles) {
                if (!wait_warp(&bars.y_empty, it & 1, abort_flag)) { ok = false; break; }
                fence_after();
                load_y(next);
            }
            // ---- output rows (b, ok)
            if (!wait_warp(&bars.out_full, it & 1, abort_flag)) { ok = false; break; }
            fence_after();
            float o[P.n2p];
#pragma unroll
            for (int aq = 0; aq < P.nacc2; ++aq) {
                const int a = P.fixed ? aq : P.nacc2 - 1 - aq;   // the small products first
                uint32_t orr[P.n2p / 16][16];
#pragma unroll
                for (int c0 = 0; c0 < P.n2p; c0 += 16)
                    tmem_ld16_async(tmem + lane_base + (uint32_t)(P.c_out + a * P.out_cols + c0), orr[c0 / 16]);
                tmem_ld_wait();
#pragma unroll
                for (int c0 = 0; c0 < P.n2p; c0 += 16) {
                    tmem_regs_ready(orr[c0 / 16]);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float x = __uint_as_float(orr[c0 / 16][i]);
                        o[c0 + i] = aq == 0 ? x : o[c0 + i] + x;
                    }
                }
            }
            fence_before();
            mbar_arrive(&bars.out_empty);
            const long long row = (long long)tile * P.rows + t;
            if (t < P.rows && row < total_rows) {
                float* dst = out + row * D2;
                if constexpr (D2 % 4 == 0) {
#pragma unroll
                    for (int i = 0; i < D2; i += 4) *(float4*)(dst + i) = make_float4(o[i], o[i + 1], o[i + 2], o[i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < D2; ++i) dst[i] = o[i];
                }
            }
        }
        if (!ok) {
            s_abort = 1;
            if (lane == 0) atomicOr(err, 32);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)P.tmem)
                     : "memory");
    }
}

}  // namespace lay

// ------------------------------------------------------------------ host side

int device_sms() {
    static std::atomic<int> cache[kMaxDevices] = {};
    int dev = 0;
    KH_CUDA(cudaGetDevice(&dev));
    const int i = dev < kMaxDevices ? dev : 0;
    int v = cache[i].load();
    if (v == 0) {
        KH_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
        cache[i].store(v);
    }
    return v;
}

namespace {

int smem_optin_max() {
    static std::atomic<int> cache[kMaxDevices] = {};
    int dev = 0;
    KH_CUDA(cudaGetDevice(&dev));
    const int i = dev < kMaxDevices ? dev : 0;
    int v = cache[i].load();
    if (v == 0) {
        KH_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        cache[i].store(v);
    }
    return v;
}

template <int D, int NPASS, bool BF>
void launch_layered(const float* Y, long long nb, int p, const float* img1, const float* img2, float* out, int* err,
                    cudaStream_t st) {
    constexpr lay::Plan P = lay::make_plan(D, NPASS, BF);
    static_assert(P.pc > 0, "no tensor-memory plan");
    constexpr int NPL = NPASS == 3 ? 2 : 1;
    const int nc = lay::n_chunks(P, p);
    const long long ntiles_ll = (nb + P.bt - 1) / P.bt;
    if (ntiles_ll > 0x7fffffffLL) fail(KH_EINVAL, "layered site contraction: too many tiles");
    const int ntiles = (int)ntiles_ll;
    if (ntiles == 0) return;
    const size_t fixed = 1024 + (size_t)lay::NSET * 128 * P.zs * 4;
    const size_t s1 = (size_t)NPL * P.b1_bytes, s2 = (size_t)NPL * P.b2_bytes;
    const size_t cap = (size_t)smem_optin_max() - 2048;   // the static barriers share the per-block limit
    int nst1 = 0, nst2 = 0;
    if (nc <= lay::MAXST && fixed + nc * (s1 + s2) <= cap) {
        nst1 = nst2 = nc;                                  // resident images
    } else {
        const int tries[6][2] = {{3, 3}, {2, 3}, {2, 2}, {1, 2}, {2, 1}, {1, 1}};
        for (auto& tr : tries) {
            const int a = tr[0] < nc ? tr[0] : nc, b = tr[1] < nc ? tr[1] : nc;
            if (fixed + a * s1 + b * s2 <= cap) {
                nst1 = a;
                nst2 = b;
                break;
            }
        }
    }
    if (nst1 == 0) fail(KH_EINVAL, "layered site contraction: shared memory too small");
    size_t smem = fixed + nst1 * s1 + nst2 * s2;
    // more than half the tensor memory: keep a second CTA off the SM (it
    // would only wait in tcgen05.alloc)
    if (P.tmem > 256 && smem <= cap / 2) smem = cap / 2 + 1024;
    static std::atomic<size_t> granted[kMaxDevices] = {};
    smem_opt_in(lay::layered_kernel<D, NPASS, BF>, smem, granted);
    const int grid = ntiles < device_sms() ? ntiles : device_sms();
    launch(lay::layered_kernel<D, NPASS, BF>, grid, lay::THREADS, smem, st, Y, nb, nc, (const uint8_t*)img1, (const uint8_t*)img2, out, ntiles, nst1, nst2, err);
}

template <int NPASS, bool BF>
void dispatch_d(const float* Y, long long nb, int D, int p, const float* img1, const float* img2, float* out,
                int* err, cudaStream_t st) {
    switch (D) {
        case 1: launch_layered<1, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 2: launch_layered<2, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 3: launch_layered<3, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 4: launch_layered<4, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 5: launch_layered<5, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 6: launch_layered<6, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 7: launch_layered<7, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        case 8: launch_layered<8, NPASS, BF>(Y, nb, p, img1, img2, out, err, st); break;
        default: fail(KH_EINVAL, "layered site contraction: D out of range");
    }
}

}  // namespace

long long layered_img1_floats(int D, int p, int npass, bool bf16) {
    const lay::Plan P = lay::make_plan(D, npass, bf16);
    if (P.pc == 0) return 0;
    return (long long)lay::n_chunks(P, p) * (npass == 3 ? 2 : 1) * P.b1_bytes / 4;
}

long long layered_img2_floats(int D, int p, int npass, bool bf16) {
    const lay::Plan P = lay::make_plan(D, npass, bf16);
    if (P.pc == 0) return 0;
    return (long long)lay::n_chunks(P, p) * (npass == 3 ? 2 : 1) * P.b2_bytes / 4;
}

void site_layered_tc(const float* Y, long long nb, int D, int p, const float* img1, const float* img2, float* out,
                     int npass, bool bf16, int* err, cudaStream_t st) {
    if (nb <= 0) return;
    if (((uintptr_t)img1 & 15) || ((uintptr_t)img2 & 15) || ((uintptr_t)out & 15) || ((uintptr_t)Y & 15))
        fail(KH_EINVAL, "layered site contraction: misaligned operand");
    if (bf16) {
        if (npass != 1) fail(KH_EINVAL, "layered site contraction: BF16 runs one pass");
        dispatch_d<1, true>(Y, nb, D, p, img1, img2, out, err, st);
    } else if (npass == 3) {
        dispatch_d<3, false>(Y, nb, D, p, img1, img2, out, err, st);
    } else {
        dispatch_d<1, false>(Y, nb, D, p, img1, img2, out, err, st);
    }
}

}  // namespace kh
