// Internal header of the eeFU GB300 library: context layout, workspace
// carving, error handling and the small generic kernels (permutation,
// strided batched GEMM on CUDA cores, reductions, casts).
#pragma once
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <atomic>
#include <cstdio>
#include <mutex>
#include <stdio.h>
#include <string.h>
#include <string>
#include <vector>

#include "../../include/eefu.h"

namespace kh {

// ------------------------------------------------------------------ errors

struct Error {
    kh_status st;
    std::string msg;
};

#define KH_CUDA(call)                                                                 \
    do {                                                                              \
        cudaError_t _e = (call);                                                      \
        if (_e != cudaSuccess) {                                                      \
            throw ::kh::Error{KH_ECUDA, std::string(#call) + ": " + cudaGetErrorString(_e) + " at " + \
                              __FILE__ + ":" + std::to_string(__LINE__)};                        \
        }                                                                             \
    } while (0)

#define KH_CHECK_LAUNCH() KH_CUDA(cudaGetLastError())
#define KH_LAUNCHED() do { KH_CUDA(cudaGetLastError()); ::kh::count_launch(); } while (0)

inline void fail(kh_status st, const std::string& m) { throw Error{st, m}; }

// number of kernels this library has launched (read by kh_launch_count);
// atomic because contexts may be driven from several host threads
extern std::atomic<unsigned long long> g_launches;
inline void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

// ------------------------------------------------------------------ launches

// Programmatic dependent launch: a kernel launched with launch() may be set up on
// the SMs while its predecessor in the stream still drains; pdl_start() at its
// top waits until that one is complete and its writes are visible, then lets
// the next one be set up.  Small moves are a chain of 70 short kernels: when it
// came in, the environment of (D, chi) = (4, 64) went from 12.84 to 11.33 ms, of
// (3, 32) in FP64 from 13.71 to 12.38, of (6, 144) from 83.4 to 81.0, the bond gradient
// from 407 to 379 us.  Where a wide kernel precedes a product of few long CTAs it
// does harm (GemmArgs::plain).  Kernels started with <<<>>> are ordered as ever, and pdl_start() returns
// at once in them.
__device__ __forceinline__ void pdl_start() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    KH_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    count_launch();
}

// TF32 head of x for the operand splits x = head + (x - head): with half = kTf32Half
// (half a unit of its last place) the nearest, with 0 the leading bits.  Rounding
// must not make a finite value infinite (infinity - infinity is NaN):
// tf32_half(m) is the half for values of magnitude m or less.  A NaN may lose its
// head and stays in the remainder.
constexpr uint32_t kTf32Half = 0x1000u;
__device__ __forceinline__ uint32_t tf32_half(float m) { return __float_as_uint(m) < 0x7f7ff000u ? kTf32Half : 0u; }
__device__ __forceinline__ float tf32_head(float x, uint32_t half) {
    return __uint_as_float((__float_as_uint(x) + half) & 0xFFFFE000u);
}

// ------------------------------------------------------------------ workspace

// Bump allocator over the caller's workspace; every block 256-byte aligned.
struct Carver {
    char* base;
    size_t cap, off;
    explicit Carver(void* b = nullptr, size_t c = 0) : base((char*)b), cap(c), off(0) {}
    template <typename T>
    T* take(size_t n) {
        size_t bytes = ((n * sizeof(T) + 255) / 256) * 256;
        size_t at = off;
        off += bytes;
        if (base == nullptr) return nullptr;          // sizing pass
        if (off > cap) fail(KH_ENOMEM, "workspace too small");
        return (T*)(base + at);
    }
};

// ------------------------------------------------------------------ permutation

constexpr int kMaxRank = 8;

// Division of 32-bit n < 2^31 by a divisor d fixed on the host: with
// l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1, q = (umulhi(n, m) + n) >> l
// (Granlund & Montgomery, "Division by invariant integers using multiplication").
struct FastDiv {
    uint32_t d, m, l;
};
inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f;
    f.d = d;
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    f.l = l;
    f.m = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
    return f;
}
__device__ __forceinline__ uint32_t fast_div(uint32_t n, const FastDiv& f) {
    return (__umulhi(n, f.m) + n) >> f.l;
}

struct PermArgs {
    int rank;
    long long total;
    long long out_dims[kMaxRank];   // output shape (row-major)
    long long in_strides[kMaxRank]; // input stride of each output axis
    FastDiv div[kMaxRank];          // output dims as fast divisors (32-bit path)
};

// out[i_0..i_{r-1}] = in[sum_j i_j * in_strides[j]]
template <typename Ti, typename To>
__global__ void permute_kernel(const Ti* __restrict__ in, To* __restrict__ out, PermArgs a) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long step = (long long)gridDim.x * blockDim.x;
    for (; idx < a.total; idx += step) {
        long long rem = idx, src = 0;
        for (int j = a.rank - 1; j >= 0; --j) {
            long long d = a.out_dims[j];
            long long i = rem % d;
            rem /= d;
            src += i * a.in_strides[j];
        }
        out[idx] = (To)in[src];
    }
}

// Same with 32-bit index arithmetic (total < 2^31): multiply-shift divisions.
template <typename Ti, typename To>
__global__ void permute32_kernel(const Ti* __restrict__ in, To* __restrict__ out, PermArgs a) {
    pdl_start();
    const uint32_t total = (uint32_t)a.total;
    const uint32_t step = gridDim.x * blockDim.x;
    for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += step) {
        uint32_t rem = idx, src = 0;
#pragma unroll
        for (int j = kMaxRank - 1; j >= 0; --j) {
            if (j < a.rank) {
                const uint32_t q = fast_div(rem, a.div[j]);
                src += (rem - q * a.div[j].d) * (uint32_t)a.in_strides[j];
                rem = q;
            }
        }
        out[idx] = (To)in[src];
    }
}

// Permutation fused with the 3xTF32 operand split: hi = the value rounded to
// nearest TF32 or cut off there, lo = value - hi (32-bit path); the permuted value itself also goes
// to out when out is not null.
static __global__ void permute_split32_kernel(const float* __restrict__ in, float* __restrict__ hi,
                                              float* __restrict__ lo, float* __restrict__ out, bool nearest, PermArgs a) {
    pdl_start();
    const uint32_t total = (uint32_t)a.total;
    const uint32_t step = gridDim.x * blockDim.x;
    for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += step) {
        uint32_t rem = idx, src = 0;
#pragma unroll
        for (int j = kMaxRank - 1; j >= 0; --j) {
            if (j < a.rank) {
                const uint32_t q = fast_div(rem, a.div[j]);
                src += (rem - q * a.div[j].d) * (uint32_t)a.in_strides[j];
                rem = q;
            }
        }
        const float v = in[src];
        const float h = tf32_head(v, nearest ? tf32_half(fabsf(v)) : 0u);
        hi[idx] = h;
        lo[idx] = v - h;
        if (out) out[idx] = v;
    }
}

// Build PermArgs from an input shape and the axis order of the output:
// out axis j is input axis order[j].
inline PermArgs make_perm(const std::vector<long long>& in_shape, const std::vector<int>& order) {
    PermArgs a;
    memset(&a, 0, sizeof(a));
    int r = (int)in_shape.size();
    if (r > kMaxRank || (int)order.size() != r) fail(KH_EINVAL, "permute rank");
    std::vector<long long> in_str(r);
    long long s = 1;
    for (int j = r - 1; j >= 0; --j) { in_str[j] = s; s *= in_shape[j]; }
    a.rank = r;
    a.total = s;
    for (int j = 0; j < r; ++j) {
        a.out_dims[j] = in_shape[order[j]];
        a.in_strides[j] = in_str[order[j]];
        if (a.out_dims[j] >= 1 && a.out_dims[j] < (1LL << 31)) a.div[j] = make_fastdiv((uint32_t)a.out_dims[j]);
    }
    return a;
}

// Let a kernel launch with `bytes` of dynamic shared memory on the current
// device: the 48 KB default covers static plus dynamic shared memory, so the
// opt-in is made when the kernel's static size plus `bytes` exceeds it; once
// per (kernel, device) and size, cache being the call site's table of the
// sizes already settled, indexed by device ordinal (the attribute is per
// device, so a context on a second GPU needs its own opt-in).  Contexts may
// live on several host threads: the settled size is read lock-free, and a
// raise is made under one lock, so the attribute only ever grows (a smaller
// request arriving second never lowers a larger grant another thread is
// about to launch with).
constexpr int kMaxDevices = 64;
inline std::mutex& smem_opt_in_mutex() {
    static std::mutex m;
    return m;
}
template <typename K>
inline void smem_opt_in(K kernel, size_t bytes, std::atomic<size_t> (&cache)[kMaxDevices]) {
    int dev = 0;
    KH_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) fail(KH_EINVAL, "device ordinal beyond 63");
    if (cache[dev].load(std::memory_order_acquire) >= bytes) return;
    std::lock_guard<std::mutex> lock(smem_opt_in_mutex());
    if (cache[dev].load(std::memory_order_relaxed) >= bytes) return;
    cudaFuncAttributes fa;
    KH_CUDA(cudaFuncGetAttributes(&fa, kernel));
    if (fa.sharedSizeBytes + bytes > 48 * 1024)
        KH_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    cache[dev].store(bytes, std::memory_order_release);
}

inline int grid_for(long long n, int block = 256) {
    long long g = (n + block - 1) / block;
    if (g > 152LL * 64) g = 152LL * 64;
    if (g < 1) g = 1;
    return (int)g;
}

// Large permutations: tiles of all the axes that make up the fastest runs (>= 16
// elements) of the input and of the output, staged in shared memory, so that
// both sides are read and written in runs.  A CTA takes G tiles at a time (about
// 2048 elements); the offsets inside a tile and the place of every output
// element in the staged tile are tables made once per CTA, the tiles' base
// offsets are computed by one thread each.  Against the element-wise kernels,
// whose strided reads fetch every sector several times: the permutations of a
// move at (D, chi) = (6, 144), 27 M floats each, went from 83 to 57 us on
// average, at (8, 144), 85 M, from 324 to 150; the split form keeps its time.
struct TileArgs {
    int ndim, nouter_dims;
    uint32_t te, nouter, group;                  // elements of a tile, tiles, tiles at a time
    FastDiv te_div;
    int tdims_in[kMaxRank], ts_in[kMaxRank];     // tile axes, slowest first in the input, and input strides
    int tdims_out[kMaxRank], ts_out[kMaxRank], tin_of_out[kMaxRank];   // in the output: output and staged strides
    FastDiv odiv[kMaxRank];                      // the other axes (slowest first)
    uint32_t os_in[kMaxRank], os_out[kMaxRank];
};
constexpr int kTileMax = 2048, kTileGroupMax = 64;

template <typename Ti, typename To, bool SPLIT>
__global__ void __launch_bounds__(256)
permute_tiled_kernel(const Ti* __restrict__ in, To* __restrict__ out, float* __restrict__ hi, float* __restrict__ lo,
                     bool nearest, TileArgs a) {
    pdl_start();
    __shared__ Ti tile[kTileMax + kTileMax / 32];
    __shared__ uint32_t off_in[kTileMax], off_out[kTileMax];
    __shared__ uint16_t place[kTileMax];
    __shared__ uint32_t base_in[kTileGroupMax], base_out[kTileGroupMax];
    const int tid = threadIdx.x;
    for (uint32_t e = tid; e < a.te; e += 256) {
        uint32_t rem = e, oi = 0;
        for (int j = a.ndim - 1; j >= 0; --j) {
            oi += (rem % a.tdims_in[j]) * a.ts_in[j];
            rem /= a.tdims_in[j];
        }
        off_in[e] = oi;
        uint32_t oo = 0, pl = 0;
        rem = e;
        for (int j = a.ndim - 1; j >= 0; --j) {
            const uint32_t x = rem % a.tdims_out[j];
            oo += x * a.ts_out[j];
            pl += x * a.tin_of_out[j];
            rem /= a.tdims_out[j];
        }
        off_out[e] = oo;
        place[e] = (uint16_t)pl;
    }
    const uint32_t step = gridDim.x * a.group, n = a.group * a.te;
    for (uint32_t t0 = blockIdx.x * a.group; t0 < a.nouter; t0 += step) {
        __syncthreads();
        if (tid < (int)a.group && t0 + tid < a.nouter) {
            uint32_t rem = t0 + tid, bi = 0, bo = 0;
            for (int j = a.nouter_dims - 1; j >= 0; --j) {
                const uint32_t q = fast_div(rem, a.odiv[j]), x = rem - q * a.odiv[j].d;
                bi += x * a.os_in[j];
                bo += x * a.os_out[j];
                rem = q;
            }
            base_in[tid] = bi;
            base_out[tid] = bo;
        }
        __syncthreads();
        const uint32_t m = min(n, (a.nouter - t0) * a.te);
        // eight loads in flight a thread (no branch around them)
        Ti v[kTileMax / 256];
#pragma unroll
        for (int q = 0; q < kTileMax / 256; ++q) {
            const uint32_t x = min((uint32_t)tid + 256u * q, m - 1), g = fast_div(x, a.te_div);
            v[q] = in[base_in[g] + off_in[x - g * a.te]];
        }
#pragma unroll
        for (int q = 0; q < kTileMax / 256; ++q) {
            const uint32_t x = tid + 256 * q;
            if (x < m) tile[x + (x >> 5)] = v[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kTileMax / 256; ++q) {
            const uint32_t x = tid + 256 * q, xc = min(x, m - 1), g = fast_div(xc, a.te_div), e = xc - g * a.te;
            const uint32_t p = g * a.te + place[e], o = base_out[g] + off_out[e];
            const Ti w = tile[p + (p >> 5)];
            if (x >= m) continue;
            if constexpr (SPLIT) {
                const float h = tf32_head(w, nearest ? tf32_half(fabsf(w)) : 0u);
                hi[o] = h;
                lo[o] = w - h;
            }
            if (!SPLIT || out) out[o] = (To)w;
        }
    }
}

// The tiled plan of a permutation, or false where it does not apply: no tile of
// 32 to 2048 elements, or a small tensor, which fits the L2 and takes the
// element-wise kernel 7.5 us at a million elements, most of it the launch.
inline bool make_tile_args(const std::vector<long long>& in_shape, const std::vector<int>& order, TileArgs& a) {
    long long total = 1;
    for (long long d : in_shape) total *= d;
    if (total < (1LL << 21) || total >= (1LL << 31)) return false;
    // axes as (size, input stride, output stride); a long fastest axis is split so
    // that only a divisor of at least 16 of it belongs to the tile
    struct Axis {
        long long n, si, so;
        bool tile;
    };
    std::vector<Axis> ax(in_shape.size());
    long long s = 1;
    for (int j = (int)in_shape.size() - 1; j >= 0; --j) {
        ax[j].n = in_shape[j];
        ax[j].si = s;
        ax[j].tile = false;
        s *= in_shape[j];
    }
    s = 1;
    for (int j = (int)order.size() - 1; j >= 0; --j) {
        ax[order[j]].so = s;
        s *= in_shape[order[j]];
    }
    auto by = [&](bool input) {
        std::vector<int> id(ax.size());
        for (size_t i = 0; i < id.size(); ++i) id[i] = (int)i;
        for (size_t i = 1; i < id.size(); ++i)          // insertion sort, fastest first
            for (size_t j = i; j > 0; --j) {
                const Axis &p = ax[id[j]], &q = ax[id[j - 1]];
                const long long sp = input ? p.si : p.so, sq = input ? q.si : q.so;
                if (sp < sq || (sp == sq && p.n < q.n)) std::swap(id[j], id[j - 1]);
            }
        return id;
    };
    for (int side = 0; side < 2; ++side) {
        long long run = 1;
        for (int i : by(side == 0)) {
            if (run >= 16) break;
            const long long need = (16 + run - 1) / run;
            if (!ax[i].tile && ax[i].n > 24) {
                long long c = need;
                while (ax[i].n % c) ++c;
                if (c < ax[i].n) {
                    ax.push_back(Axis{ax[i].n / c, ax[i].si * c, ax[i].so * c, false});
                    ax[i].n = c;
                }
            }
            ax[i].tile = true;
            run *= ax[i].n;
        }
    }
    if ((int)ax.size() > kMaxRank) return false;
    memset(&a, 0, sizeof(a));
    const std::vector<int> fi = by(true), fo = by(false);
    std::vector<long long> staged(ax.size(), 0);         // stride of a tile axis in the staged tile
    long long te = 1;
    for (int i : fi)
        if (ax[i].tile) {
            staged[i] = te;
            te *= ax[i].n;
        }
    if (te < 32 || te > kTileMax) return false;
    int d = 0;
    for (int q = (int)fi.size() - 1; q >= 0; --q)
        if (ax[fi[q]].tile) {
            a.tdims_in[d] = (int)ax[fi[q]].n;
            a.ts_in[d++] = (int)ax[fi[q]].si;
        }
    a.ndim = d;
    d = 0;
    for (int q = (int)fo.size() - 1; q >= 0; --q)
        if (ax[fo[q]].tile) {
            a.tdims_out[d] = (int)ax[fo[q]].n;
            a.ts_out[d] = (int)ax[fo[q]].so;
            a.tin_of_out[d++] = (int)staged[fo[q]];
        }
    // the other axes, slowest in the output first: neighbouring tiles of a group write neighbouring runs
    d = 0;
    for (int q = (int)fo.size() - 1; q >= 0; --q)
        if (!ax[fo[q]].tile) {
            a.odiv[d] = make_fastdiv((uint32_t)ax[fo[q]].n);
            a.os_in[d] = (uint32_t)ax[fo[q]].si;
            a.os_out[d++] = (uint32_t)ax[fo[q]].so;
        }
    a.nouter_dims = d;
    a.te = (uint32_t)te;
    a.te_div = make_fastdiv(a.te);
    a.nouter = (uint32_t)(total / te);
    a.group = (uint32_t)(kTileMax / te);
    if (a.group > kTileGroupMax) a.group = kTileGroupMax;
    return true;
}

inline int tile_grid(const TileArgs& a) {
    const long long g = ((long long)a.nouter + a.group - 1) / a.group;
    return (int)(g < 152 * 5 ? g : 152 * 5);             // about five CTAs' shared memory per SM
}

inline void permute_split(const float* in, float* hi, float* lo, const std::vector<long long>& in_shape,
                          const std::vector<int>& order, cudaStream_t st, float* out = nullptr, bool nearest = true) {
    PermArgs a = make_perm(in_shape, order);
    if (a.total <= 0) return;
    if (a.total >= (1LL << 31)) fail(KH_EINVAL, "permute_split: tensor too large");
    TileArgs t;
    if (make_tile_args(in_shape, order, t)) {
        launch(permute_tiled_kernel<float, float, true>, tile_grid(t), 256, 0, st, in, out, hi, lo, nearest, t);
        return;
    }
    launch(permute_split32_kernel, grid_for(a.total), 256, 0, st, in, hi, lo, out, nearest, a);
}

template <typename Ti, typename To>
inline void permute(const Ti* in, To* out, const std::vector<long long>& in_shape,
                    const std::vector<int>& order, cudaStream_t st) {
    PermArgs a = make_perm(in_shape, order);
    if (a.total <= 0) return;
    TileArgs t;
    if (make_tile_args(in_shape, order, t)) {
        launch(permute_tiled_kernel<Ti, To, false>, tile_grid(t), 256, 0, st, in, out, nullptr, nullptr, false, t);
        return;
    }
    if (a.total < (1LL << 31)) {
        launch(permute32_kernel<Ti, To>, grid_for(a.total), 256, 0, st, in, out, a);
        return;
    }
    permute_kernel<Ti, To><<<grid_for(a.total), 256, 0, st>>>(in, out, a);
    KH_LAUNCHED();
}

template <typename Ti, typename To>
__global__ void cast_kernel(const Ti* __restrict__ in, To* __restrict__ out, long long n) {
    pdl_start();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long step = (long long)gridDim.x * blockDim.x;
    for (; i < n; i += step) out[i] = (To)in[i];
}

template <typename Ti, typename To>
inline void cast(const Ti* in, To* out, long long n, cudaStream_t st) {
    launch(cast_kernel<Ti, To>, grid_for(n), 256, 0, st, in, out, n);
}

// ------------------------------------------------------------------ SIMT GEMM

// C[b](m,n) = alpha * colscale[n] * sum_k A[b](m,k) B[b](k,n) + beta * C[b](m,n)
// with arbitrary element strides.  CUDA-core FMA in T.
template <typename T>
struct GemmArgs {
    int M, N, K, batch;
    const T* A; long long sAm, sAk, sAb;
    const T* B; long long sBk, sBn, sBb;
    T* C; long long sCm, sCn, sCb;
    T alpha, beta;
    const T* colscale;   // nullable, length N
    T* sk = nullptr;     // optional split-K scratch (for few output tiles and long K)
    long long sk_elems = 0;
    // started without programmatic launch: where a kernel of many CTAs comes before,
    // the CTAs of a product that does not fill the GPU would be set up in pairs on
    // the SMs that drain first, and stay there (bond metric at (5, 144): 100 CTAs of
    // 1.1 ms; the gradient took 2.61 ms so, 1.87 with an ordinary launch, 0.90 and
    // 0.57 at (5, 64))
    bool plain = false;
};

constexpr int GT_K = 16;

// Tile BM x BN per CTA, each of the 256 threads computes TM x TN outputs
// strided by (BM/TM, BN/TN) so that shared-memory reads are conflict-free.
template <typename T, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(256) gemm_simt_kernel(GemmArgs<T> g) {
    pdl_start();
    static_assert((BM / TM) * (BN / TN) == 256, "256 threads");
    constexpr int RX = BN / TN;                    // threads along N
    __shared__ T As[GT_K][BM + 1];
    __shared__ T Bs[GT_K][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid % RX, ty = tid / RX;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const long long b = blockIdx.z;
    const T* A = g.A + b * g.sAb;
    const T* B = g.B + b * g.sBb;
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    const bool a_kfast = (g.sAk == 1);
    const bool b_nfast = (g.sBn == 1);
    // register double buffering: the next K tile's global loads are issued
    // before the current tile's FMAs
    constexpr int NA = BM * GT_K / 256, NB = BN * GT_K / 256;
    static_assert(NA * 256 == BM * GT_K && NB * 256 == BN * GT_K, "tile/thread mismatch");
    T ra[NA], rb[NB];
    auto load_tiles = [&](int k0) {
#pragma unroll
        for (int t = 0; t < NA; ++t) {
            const int e = tid + 256 * t;
            int mm, kk;
            if (a_kfast) { mm = e / GT_K; kk = e % GT_K; } else { mm = e % BM; kk = e / BM; }
            const int gm = m0 + mm, gk = k0 + kk;
            ra[t] = (gm < g.M && gk < g.K) ? A[gm * g.sAm + gk * g.sAk] : T(0);
        }
#pragma unroll
        for (int t = 0; t < NB; ++t) {
            const int e = tid + 256 * t;
            int nn, kb;
            if (b_nfast) { nn = e % BN; kb = e / BN; } else { nn = e / GT_K; kb = e % GT_K; }
            const int gn = n0 + nn, gkb = k0 + kb;
            rb[t] = (gn < g.N && gkb < g.K) ? B[gkb * g.sBk + gn * g.sBn] : T(0);
        }
    };
    load_tiles(0);
    for (int k0 = 0; k0 < g.K; k0 += GT_K) {
#pragma unroll
        for (int t = 0; t < NA; ++t) {
            const int e = tid + 256 * t;
            int mm, kk;
            if (a_kfast) { mm = e / GT_K; kk = e % GT_K; } else { mm = e % BM; kk = e / BM; }
            As[kk][mm] = ra[t];
        }
#pragma unroll
        for (int t = 0; t < NB; ++t) {
            const int e = tid + 256 * t;
            int nn, kb;
            if (b_nfast) { nn = e % BN; kb = e / BN; } else { nn = e / GT_K; kb = e % GT_K; }
            Bs[kb][nn] = rb[t];
        }
        __syncthreads();
        if (k0 + GT_K < g.K) load_tiles(k0 + GT_K);
#pragma unroll
        for (int kk = 0; kk < GT_K; ++kk) {
            T a[TM], bb[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + (BM / TM) * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx + RX * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
        }
        __syncthreads();
    }
    T* C = g.C + b * g.sCb;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int gm = m0 + ty + (BM / TM) * i;
        if (gm >= g.M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            int gn = n0 + tx + RX * j;
            if (gn >= g.N) continue;
            T v = g.alpha * acc[i][j];
            if (g.colscale) v *= g.colscale[gn];
            T* dst = C + gm * g.sCm + gn * g.sCn;
            if (g.beta != T(0)) v += g.beta * (*dst);
            *dst = v;
        }
    }
}

// FP64 GEMM.  The SM's FP64 pipe (a few FMAs per clock) is the bound, not shared
// memory or L2: even an 8 x 8 tile asks for some 10 bytes per clock and SM.
// What costs time is an uneven spread over the SMs, so the tiles are small:
// 8 x 8 outputs per CTA (one per thread and K group) until there are eight
// 16 x 16 tiles per SM, from where the larger tile leaves less to fetch.  KG
// groups of threads split each K chunk; their sums are joined in shared
// memory in a fixed order.  288 x 48 x 288 (n, k of D = 3, chi = 32): 7.3 us, with
// 16 x 128 tiles 57; 288^3: 18 us (2.7 TFLOP/s), with 64 x 64 tiles 79.
template <int TB, int TT>
__global__ void __launch_bounds__(128) gemm_f64_kernel(GemmArgs<double> g) {
    pdl_start();
    constexpr int RX = TB / TT;                    // threads along N of one K group
    constexpr int GT = RX * RX;                    // threads of one K group
    constexpr int KG = 128 / GT;
    constexpr int KC = 32;                         // K chunk staged at a time
    static_assert(KC % KG == 0 && (TB * KC) % 128 == 0, "tile/thread mismatch");
    constexpr int NL = TB * KC / 128;
    __shared__ double As[KC][TB + 1], Bs[KC][TB + 1];
    __shared__ double red[KG > 1 ? (KG - 1) * TB * TB : 1];
    const int tid = threadIdx.x, kg = tid / GT, t = tid % GT, tx = t % RX, ty = t / RX;
    const int nt = (g.N + TB - 1) / TB;            // tiles along N; the tiles lie on grid.x, whose limit is 2^31
    const int m0 = (int)(blockIdx.x / nt) * TB, n0 = (int)(blockIdx.x % nt) * TB;
    const double* A = g.A + (long long)blockIdx.z * g.sAb;
    const double* B = g.B + (long long)blockIdx.z * g.sBb;
    const bool a_kfast = g.sAk == 1, b_nfast = g.sBn == 1;
    double acc[TT][TT], ra[NL], rb[NL];
#pragma unroll
    for (int i = 0; i < TT; ++i)
#pragma unroll
        for (int j = 0; j < TT; ++j) acc[i][j] = 0.0;
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < NL; ++q) {
            const int e = tid + 128 * q;
            const int ma = a_kfast ? e / KC : e % TB, ka = a_kfast ? e % KC : e / TB;
            const int nb = b_nfast ? e % TB : e / KC, kb = b_nfast ? e / TB : e % KC;
            ra[q] = (m0 + ma < g.M && k0 + ka < g.K) ? A[(m0 + ma) * g.sAm + (k0 + ka) * g.sAk] : 0.0;
            rb[q] = (n0 + nb < g.N && k0 + kb < g.K) ? B[(k0 + kb) * g.sBk + (n0 + nb) * g.sBn] : 0.0;
        }
    };
    load(0);
    for (int k0 = 0; k0 < g.K; k0 += KC) {
#pragma unroll
        for (int q = 0; q < NL; ++q) {
            const int e = tid + 128 * q;
            As[a_kfast ? e % KC : e / TB][a_kfast ? e / KC : e % TB] = ra[q];
            Bs[b_nfast ? e / TB : e % KC][b_nfast ? e % TB : e / KC] = rb[q];
        }
        __syncthreads();
        if (k0 + KC < g.K) load(k0 + KC);
        const int kn = min(KC, g.K - k0);
#pragma unroll 4
        for (int kk = kg; kk < kn; kk += KG) {
            double a[TT], b[TT];
#pragma unroll
            for (int i = 0; i < TT; ++i) a[i] = As[kk][ty + RX * i];
#pragma unroll
            for (int j = 0; j < TT; ++j) b[j] = Bs[kk][tx + RX * j];
#pragma unroll
            for (int i = 0; i < TT; ++i)
#pragma unroll
                for (int j = 0; j < TT; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    if (KG > 1) {
        if (kg > 0)
#pragma unroll
            for (int i = 0; i < TT; ++i)
#pragma unroll
                for (int j = 0; j < TT; ++j) red[(kg - 1) * TB * TB + (i * TT + j) * GT + t] = acc[i][j];
        __syncthreads();
        if (kg > 0) return;
#pragma unroll
        for (int q = 0; q < KG - 1; ++q)
#pragma unroll
            for (int i = 0; i < TT; ++i)
#pragma unroll
                for (int j = 0; j < TT; ++j) acc[i][j] += red[q * TB * TB + (i * TT + j) * GT + t];
    }
    double* C = g.C + (long long)blockIdx.z * g.sCb;
#pragma unroll
    for (int i = 0; i < TT; ++i) {
        const int gm = m0 + ty + RX * i;
        if (gm >= g.M) continue;
#pragma unroll
        for (int j = 0; j < TT; ++j) {
            const int gn = n0 + tx + RX * j;
            if (gn >= g.N) continue;
            double v = g.alpha * acc[i][j];
            if (g.colscale) v *= g.colscale[gn];
            double* dst = C + gm * g.sCm + gn * g.sCn;
            if (g.beta != 0.0) v += g.beta * (*dst);
            *dst = v;
        }
    }
}

inline void gemm_f64(const GemmArgs<double>& g, cudaStream_t st) {
    auto tiles = [&](int tb) { return (long long)((g.M + tb - 1) / tb) * ((g.N + tb - 1) / tb) * g.batch; };
    const bool small = tiles(16) < 8LL * 152;
    const int tb = small ? 8 : 16;
    const long long nt = (long long)((g.M + tb - 1) / tb) * ((g.N + tb - 1) / tb);
    if (nt > 0x7fffffffLL) fail(KH_EINVAL, "gemm too large");
    const dim3 grid((unsigned)nt, 1, g.batch);
    if (small) launch(gemm_f64_kernel<8, 1>, grid, 128, 0, st, g);
    else launch(gemm_f64_kernel<16, 2>, grid, 128, 0, st, g);
}

template <typename T, int BM, int BN, int TM, int TN>
inline void gemm_launch(const GemmArgs<T>& g, cudaStream_t st) {
    dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
    if (grid.y > 65535) fail(KH_EINVAL, "gemm M too large");
    if (g.plain && (long long)grid.x * grid.y * grid.z < 2 * 152) {
        gemm_simt_kernel<T, BM, BN, TM, TN><<<grid, 256, 0, st>>>(g);
        KH_LAUNCHED();
        return;
    }
    launch(gemm_simt_kernel<T, BM, BN, TM, TN>, grid, 256, 0, st, g);
}

// out[i] = alpha * colscale[col] * sum_s part[s][i] + beta * out   (split-K reduction)
template <typename T>
__global__ void splitk_reduce_kernel(const T* __restrict__ part, int splits, int M, int N, T* C, long long sCm,
                                     long long sCn, T alpha, T beta, const T* colscale) {
    pdl_start();
    long long tot = (long long)M * N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
         i += (long long)gridDim.x * blockDim.x) {
        T acc = T(0);
        for (int s = 0; s < splits; ++s) acc += part[s * tot + i];
        int m = (int)(i / N), n = (int)(i % N);
        T v = alpha * acc;
        if (colscale) v *= colscale[n];
        T* dst = C + m * sCm + n * sCn;
        if (beta != T(0)) v += beta * (*dst);
        *dst = v;
    }
}

template <typename T>
inline void gemm_dispatch(const GemmArgs<T>& g, cudaStream_t st) {
    const long long tiles64 = (long long)((g.M + 63) / 64) * ((g.N + 63) / 64) * g.batch;
    if (g.M <= 16 && g.N <= 16) gemm_launch<T, 16, 16, 1, 1>(g, st);
    else if (g.N <= 16) gemm_launch<T, 128, 16, 2, 4>(g, st);
    else if (g.M <= 16) gemm_launch<T, 16, 128, 4, 2>(g, st);
    else if (g.N <= 128 && tiles64 < 76) gemm_launch<T, 16, 128, 4, 2>(g, st);   // few 64x64 tiles: more, thinner CTAs
    else gemm_launch<T, 64, 64, 4, 4>(g, st);
}

// Few output tiles and a long K (FP32): the partial products of K split over
// CTAs go to the scratch as parts of M x N each, and their number is returned;
// 0 where K is not split (nothing is launched).
template <typename T>
inline int gemm_parts(const GemmArgs<T>& g, cudaStream_t st) {
    const long long tiles = (long long)((g.M + 63) / 64) * ((g.N + 63) / 64);
    if (sizeof(T) == 8 || g.batch != 1 || !g.sk || tiles >= 76 || g.K < 256) return 0;
    int splits = (int)((304 + tiles - 1) / tiles);   // about two CTAs per SM
    int maxs = g.K / 128;
    if (splits > maxs) splits = maxs;
    if (splits > 32) splits = 32;
    const long long mn = (long long)g.M * g.N;
    if (splits < 2 || splits * mn > g.sk_elems) return 0;
    const int kchunk = ((g.K + splits - 1) / splits + GT_K - 1) / GT_K * GT_K;
    splits = (g.K + kchunk - 1) / kchunk;
    GemmArgs<T> p = g;
    p.K = kchunk;
    p.batch = splits;
    p.sAb = kchunk * g.sAk;            // batch b = K range [b*kchunk, ...)
    p.sBb = kchunk * g.sBk;
    p.C = g.sk; p.sCm = g.N; p.sCn = 1; p.sCb = mn;
    p.alpha = T(1); p.beta = T(0); p.colscale = nullptr; p.sk = nullptr;
    // the last chunk may overrun K: handled by a separate launch with the remainder
    const int last = g.K - (splits - 1) * kchunk;
    if (last == kchunk) {
        gemm_dispatch<T>(p, st);
    } else {
        p.batch = splits - 1;
        gemm_dispatch<T>(p, st);
        GemmArgs<T> r = p;
        r.batch = 1; r.K = last;
        r.A = g.A + (long long)(splits - 1) * kchunk * g.sAk;
        r.B = g.B + (long long)(splits - 1) * kchunk * g.sBk;
        r.C = g.sk + (long long)(splits - 1) * mn;
        gemm_dispatch<T>(r, st);
    }
    return splits;
}

template <typename T>
inline void gemm(const GemmArgs<T>& g, cudaStream_t st) {
    if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return;
    if (g.batch > 65535) fail(KH_EINVAL, "gemm batch > 65535");
    if constexpr (sizeof(T) == 8) {
        gemm_f64(g, st);
    } else {
        const int splits = gemm_parts<T>(g, st);     // joined in a fixed order (deterministic)
        if (splits) {
            launch(splitk_reduce_kernel<T>, grid_for((long long)g.M * g.N), 256, 0, st,
                g.sk, splits, g.M, g.N, g.C, g.sCm, g.sCn, g.alpha, g.beta, g.colscale);
            return;
        }
        gemm_dispatch<T>(g, st);
    }
}

// Arguments of the plain row-major C(MxN) = A(MxK) B(KxN); transposes by flags.
template <typename T>
inline GemmArgs<T> rm_args(int M, int N, int K, const T* A, bool tA, const T* B, bool tB, T* C) {
    GemmArgs<T> g;
    g.M = M; g.N = N; g.K = K; g.batch = 1;
    g.A = A; g.sAm = tA ? 1 : K; g.sAk = tA ? M : 1; g.sAb = 0;
    g.B = B; g.sBk = tB ? 1 : N; g.sBn = tB ? K : 1; g.sBb = 0;
    g.C = C; g.sCm = N; g.sCn = 1; g.sCb = 0;
    g.alpha = T(1); g.beta = T(0); g.colscale = nullptr;
    return g;
}

// Plain row-major C(MxN) = A(MxK) B(KxN) [+beta C]; transposes by flags.
template <typename T>
inline void gemm_rm(int M, int N, int K, const T* A, bool tA, const T* B, bool tB, T* C,
                    cudaStream_t st, T alpha = T(1), T beta = T(0), const T* colscale = nullptr,
                    T* sk = nullptr, long long sk_elems = 0, bool plain = false) {
    GemmArgs<T> g = rm_args<T>(M, N, K, A, tA, B, tB, C);
    g.sk = sk;
    g.sk_elems = sk_elems;
    g.plain = plain;
    g.alpha = alpha; g.beta = beta; g.colscale = colscale;
    gemm(g, st);
}

// ------------------------------------------------------------------ reductions

// FP32 <-> FP64 conversions in integer arithmetic (the conversion instructions
// issue on the narrow FP64 pipe), without a branch.  Subnormal FP32 values pass
// through a scaling by 2^64; d2f rounds to nearest even, subnormal results up to
// one more rounding on the way.  d2f_flush makes those zero, for values that count
// next to normal ones only.
__device__ __forceinline__ double f2d(float x) {
    const bool sub = (__float_as_uint(x) & 0x7f800000u) == 0;
    const uint32_t u = __float_as_uint(sub ? x * 0x1p64f : x), e = u & 0x7f800000u;
    const uint32_t up = e == 0x7f800000u ? 0x70000000u : (sub ? 0x34000000u : 0x38000000u);
    const uint32_t hi = (u & 0x80000000u) | (e ? ((u & 0x7fffffffu) >> 3) + up : 0u);
    return __hiloint2double((int)hi, e ? (int)(u << 29) : 0);
}
__device__ __forceinline__ double f2d(double x) { return x; }
__device__ __forceinline__ float d2f_flush(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t sign = hi & 0x80000000u, mag = hi & 0x7fffffffu;
    const uint32_t r = ((mag - 0x38000000u) << 3) | (lo >> 29), rem = lo & 0x1fffffffu;
    uint32_t v = r + ((rem > 0x10000000u || (rem == 0x10000000u && (r & 1u))) ? 1u : 0u);
    const bool nan = mag > 0x7ff00000u || (mag == 0x7ff00000u && lo != 0u);
    v = mag >= 0x47f00000u ? (nan ? 0x7fc00000u : 0x7f800000u) : v;     // 2^128 and more, infinity, NaN
    v = mag < 0x38100000u ? 0u : v;
    return __uint_as_float(sign | v);
}
__device__ __forceinline__ float d2f(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const bool sub = (hi & 0x7fffffffu) < 0x38100000u;                  // below 2^-126
    const float y = d2f_flush(__hiloint2double((int)(sub ? hi + 0x04000000u : hi), __double2loint(x)));
    return sub ? y * 0x1p-64f : y;
}

// out[0] = sum x^2 (FP64 accumulate), one atomic per block; launch it on a
// grid of a few blocks per SM (sumsq_grid): one atomic per element block
// would serialise thousands of FP64 atomics on one address
template <typename T>
__global__ void sumsq_kernel(const T* __restrict__ x, long long n, double* out) {
    pdl_start();
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        double v = f2d(x[i]);
        s += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double red[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = s;
    __syncthreads();
    if (w == 0) {
        s = (lane < (int)(blockDim.x >> 5)) ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) atomicAdd(out, s);
    }
}

// FP64 reciprocal, reciprocal square root and square root by Newton-Raphson
// iteration from the FP32 hardware estimates: each step squares the relative
// error (reciprocal: y <- y + y (1 - x y); reciprocal square root:
// y <- y (3/2 - (x/2) y^2)), so two steps take the ~2^-23 estimate below FP64
// rounding (a few ulp).  FP64 division and square root issue as long
// dependent sequences on GB300's narrow FP64 pipe; these take four or five
// FP64 FMAs.  Arguments outside the FP32 normal range use the IEEE operation.
__device__ __forceinline__ double rcp_nr(double x) {
    const float ax = fabsf((float)x);
    if (!(ax > 1e-30f && ax < 1e30f)) return 1.0 / x;
    double y = (double)__frcp_rn((float)x);
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}
__device__ __forceinline__ double rsqrt_nr(double x) {      // x > 0
    const float xf = (float)x;
    if (!(xf > 1e-30f && xf < 1e30f)) return 1.0 / sqrt(x);
    double y = (double)rsqrtf(xf);
    const double h = 0.5 * x;
    y = y * fma(-h * y, y, 1.5);
    return y * fma(-h * y, y, 1.5);
}
__device__ __forceinline__ double sqrt_nr(double x) {       // x >= 0
    const float xf = (float)x;
    if (!(xf > 1e-30f && xf < 1e30f)) return sqrt(x);
    const double r = rsqrt_nr(x);
    const double s = x * r;
    return fma(fma(-s, s, x), 0.5 * r, s);                   // s + (x - s^2) / (2 sqrt x)
}

inline int sumsq_grid(long long n) {
    long long g = (n + 255) / 256;
    return (int)(g < 304 ? (g < 1 ? 1 : g) : 304);
}

}  // namespace kh
