// Row-block kernels of the projector's subspace iteration for small bases (n x k
// blocks with k <= 96 and a few thousand rows, FP32).
//
// At D = 4, chi = 64 (n = 1024, k = 80) an orthonormalisation was nine launches of
// 3 to 9 us each, all of them launch and memory latency: K-split reduction, Gram,
// factor, product, Gram, factor, product and two clears.  Here every pass over
// the n x k block is one launch that does all it can with a block of 32 rows in
// shared memory: it forms the rows (sum of the K split's parts, product with a
// k x k factor, projection off the live columns) and adds their Gram matrix.
// The Gram sums are those of gram_kernel (FP32 over 16 rows, then FP64).
// At n = 1024, k = 80 the passes take 12 to 16 us each, where the launches that
// they replace took 3 to 9 us each and twice as many gaps: the environment of
// (D, chi) = (4, 64) went from 13.46 to 12.84 ms, its launches from 1387 to 1099.  (In
// the fixed order of make_dims the warm start's passes, rows_split and
// rows_project, give way to FP32 products, whose rounding is kept: 1179.)
#include "engine.cuh"

namespace kh {

namespace {

constexpr int kRows = 32;                // rows per CTA: fewer would double the FP64 atomics of the Gram sums

// rows of a (n x k) block into a padded tile (zero outside)
template <int KT>
__device__ __forceinline__ void load_rows(const float* __restrict__ Y, int r0, int n, int k, float (*t)[16 * KT]) {
    constexpr int KP = 16 * KT, PER = kRows * KP / 256;
    float v[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int e = threadIdx.x + 256 * q, r = e / KP, c = e % KP;
        const float x = Y[(long long)min(r0 + r, n - 1) * k + min(c, k - 1)];
        v[q] = (r0 + r < n && c < k) ? x : 0.f;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int e = threadIdx.x + 256 * q;
        t[e / KP][e % KP] = v[q];
    }
}

// a k x k factor (FP32, or FP64 rounded) into shared memory, zero padded
template <int KT, typename TX>
__device__ __forceinline__ void load_factor(const TX* __restrict__ X, int k, float (*s)[16 * KT]) {
    constexpr int KP = 16 * KT, PER = KP * KP / 256;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int e = threadIdx.x + 256 * q, r = e / KP, c = e % KP;
        const TX x = X[(long long)min(r, k - 1) * k + min(c, k - 1)];
        float f;
        if constexpr (sizeof(TX) == 8) f = d2f(x);
        else f = x;
        s[r][c] = (r < k && c < k) ? f : 0.f;
    }
}

// acc[i][b] = sum_m t[ty + 16 i][m] s[m][tx + 16 b]
template <int KT>
__device__ __forceinline__ void multiply(const float (*t)[16 * KT], const float (*s)[16 * KT], int k, int tx, int ty,
                                         float (&acc)[2][KT]) {
#pragma unroll
    for (int b = 0; b < KT; ++b) acc[0][b] = acc[1][b] = 0.f;
#pragma unroll 4
    for (int m = 0; m < k; ++m) {
        const float y0 = t[ty][m], y1 = t[ty + 16][m];
#pragma unroll
        for (int b = 0; b < KT; ++b) {
            const float x = s[m][tx + 16 * b];
            acc[0][b] = fmaf(y0, x, acc[0][b]);
            acc[1][b] = fmaf(y1, x, acc[1][b]);
        }
    }
}

// G += A^T B of the two tiles' rows
template <int KT>
__device__ __forceinline__ void add_gram(const float (*A)[16 * KT], const float (*B)[16 * KT], int k, int ti, int tj,
                                         double* __restrict__ G) {
    float s0[KT][KT], acc[KT][KT];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int a = 0; a < KT; ++a)
#pragma unroll
            for (int b = 0; b < KT; ++b) acc[a][b] = 0.f;
#pragma unroll 4
        for (int r = 16 * h; r < 16 * h + 16; ++r) {
            float x[KT], y[KT];
#pragma unroll
            for (int a = 0; a < KT; ++a) {
                x[a] = A[r][ti + 16 * a];
                y[a] = B[r][tj + 16 * a];
            }
#pragma unroll
            for (int a = 0; a < KT; ++a)
#pragma unroll
                for (int b = 0; b < KT; ++b) acc[a][b] = fmaf(x[a], y[b], acc[a][b]);
        }
        if (h == 0) {
#pragma unroll
            for (int a = 0; a < KT; ++a)
#pragma unroll
                for (int b = 0; b < KT; ++b) s0[a][b] = acc[a][b];
        }
    }
#pragma unroll
    for (int a = 0; a < KT; ++a)
#pragma unroll
        for (int b = 0; b < KT; ++b) {
            const int i = ti + 16 * a, j = tj + 16 * b;
            if (i < k && j < k) atomicAdd(&G[i * k + j], f2d(s0[a][b]) + f2d(acc[a][b]));
        }
}

// Y = sum of the K split's parts (n x k each, in order; not stored when Y is
// null), and its Gram matrix into G
template <int KT>
__global__ void __launch_bounds__(256)
rows_reduce_kernel(const float* __restrict__ part, int splits, int n, int k, float* __restrict__ Y,
                   double* __restrict__ G) {
    pdl_start();
    constexpr int KP = 16 * KT, PER = kRows * KP / 256;
    __shared__ float t[kRows][KP];
    const int tid = threadIdx.x, r0 = blockIdx.x * kRows;
    const long long stride = (long long)n * k;
    float v[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) v[q] = 0.f;
    for (int s = 0; s < splits; ++s) {
        const float* p = part + s * stride;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int e = tid + 256 * q, r = e / KP, c = e % KP;
            v[q] += p[(long long)min(r0 + r, n - 1) * k + min(c, k - 1)];
        }
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int e = tid + 256 * q, r = e / KP, c = e % KP;
        const bool in = r0 + r < n && c < k;
        t[r][c] = in ? v[q] : 0.f;
        if (in && Y) Y[(long long)(r0 + r) * k + c] = v[q];
    }
    __syncthreads();
    add_gram<KT>(t, t, k, tid >> 4, tid & 15, G);
}

struct RowsOperands {
    const float* Y[2];
    const float* X[2];
    float* Q[2];
};

// Q = Y X for one or (blockIdx.y) two pairs, with the Gram matrix of Q into G when given
template <int KT>
__global__ void __launch_bounds__(256)
rows_apply_kernel(RowsOperands o, int n, int k, double* __restrict__ G) {
    pdl_start();
    constexpr int KP = 16 * KT;
    extern __shared__ float rows_smem[];
    float(*t)[KP] = reinterpret_cast<float(*)[KP]>(rows_smem);
    float(*s)[KP] = t + kRows;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, r0 = blockIdx.x * kRows;
    const float *Y = o.Y[blockIdx.y], *X = o.X[blockIdx.y];
    float* Q = o.Q[blockIdx.y];
    load_rows<KT>(Y, r0, n, k, t);
    load_factor<KT>(X, k, s);
    __syncthreads();
    float acc[2][KT];
    multiply<KT>(t, s, k, tx, ty, acc);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int b = 0; b < KT; ++b) {
            const int r = ty + 16 * i, c = tx + 16 * b;
            t[r][c] = acc[i][b];                     // zero in the padding: so are Y's rows and X's columns there
            if (r0 + r < n && c < k) Q[(long long)(r0 + r) * k + c] = acc[i][b];
        }
    if (G) {
        __syncthreads();
        add_gram<KT>(t, t, k, ty, tx, G);
    }
}

// Warm basis: live columns to Vl (dead ones zero), random vectors in the dead
// columns of R (live ones zero), G += Vl^T R.
template <int KT>
__global__ void __launch_bounds__(256)
rows_split_kernel(const float* __restrict__ Vw, const int* __restrict__ live, int n, int k, float* __restrict__ Vl,
                  float* __restrict__ R, uint64_t seed, uint64_t stream, double* __restrict__ G) {
    pdl_start();
    constexpr int KP = 16 * KT, PER = kRows * KP / 256;
    __shared__ float tv[kRows][KP], tr[kRows][KP];
    const int tid = threadIdx.x, r0 = blockIdx.x * kRows;
    load_rows<KT>(Vw, r0, n, k, tv);
#pragma unroll
    for (int q = 0; q < PER; ++q) {                  // a thread's own elements: no barrier in between
        const int e = tid + 256 * q, r = e / KP, c = e % KP;
        const bool in = r0 + r < n && c < k, lv = in && live[c] != 0;
        const long long i = (long long)(r0 + r) * k + c;
        const float x = lv ? tv[r][c] : 0.f;
        const float y = in && !lv ? (float)rnd_uniform(seed, stream, (uint64_t)i) : 0.f;
        tv[r][c] = x;
        tr[r][c] = y;
        if (in) {
            Vl[i] = x;
            R[i] = y;
        }
    }
    __syncthreads();
    add_gram<KT>(tv, tr, k, tid >> 4, tid & 15, G);
}

// R <- R - Vl C with C = Vl^T R as accumulated in FP64 (rounded to FP32): the
// first time with G += Vl^T R of the new R; the second time (G null) R <- Vl + R.
template <int KT>
__global__ void __launch_bounds__(256)
rows_project_kernel(const float* __restrict__ Vl, const double* __restrict__ C, int n, int k, float* __restrict__ R,
                    double* __restrict__ G) {
    pdl_start();
    constexpr int KP = 16 * KT;
    extern __shared__ float rows_smem[];
    float(*t)[KP] = reinterpret_cast<float(*)[KP]>(rows_smem);
    float(*tr)[KP] = t + kRows;
    float(*s)[KP] = tr + kRows;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, r0 = blockIdx.x * kRows;
    load_rows<KT>(Vl, r0, n, k, t);
    load_rows<KT>(R, r0, n, k, tr);
    load_factor<KT>(C, k, s);
    __syncthreads();
    float acc[2][KT];
    multiply<KT>(t, s, k, tx, ty, acc);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int b = 0; b < KT; ++b) {
            const int r = ty + 16 * i, c = tx + 16 * b;
            const float x = tr[r][c] - acc[i][b];
            tr[r][c] = x;                            // this thread's own elements
            if (r0 + r < n && c < k) R[(long long)(r0 + r) * k + c] = G ? x : t[r][c] + x;
        }
    if (G) {
        __syncthreads();
        add_gram<KT>(t, tr, k, ty, tx, G);
    }
}

}  // namespace

#define KH_ROWS(KT)                                                                                                    \
    case KT: KH_ROWS_CALL(KT); break;
#define KH_ROWS_SWITCH                                                                                                 \
    switch ((k + 15) / 16) {                                                                                           \
        KH_ROWS(1) KH_ROWS(2) KH_ROWS(3) KH_ROWS(4) KH_ROWS(5) KH_ROWS(6) default : fail(KH_EINVAL, "rows: k > 96");   \
    }

void rows_reduce(const float* part, int splits, int n, int k, float* Y, double* G, cudaStream_t st) {
    const int grid = (n + kRows - 1) / kRows;
#define KH_ROWS_CALL(KT) launch(rows_reduce_kernel<KT>, grid, 256, 0, st, part, splits, n, k, Y, G)
    KH_ROWS_SWITCH
#undef KH_ROWS_CALL
}

void rows_apply(const float* Y, const float* X, int n, int k, float* Q, double* G, cudaStream_t st, const float* Y2,
                const float* X2, float* Q2) {
    const dim3 grid((n + kRows - 1) / kRows, Q2 ? 2 : 1);
    const RowsOperands o{{Y, Y2}, {X, X2}, {Q, Q2}};
#define KH_ROWS_CALL(KT)                                                              \
    {                                                                                 \
        constexpr size_t sm = sizeof(float) * 16 * KT * (kRows + 16 * KT);            \
        static std::atomic<size_t> granted[kMaxDevices] = {};                         \
        smem_opt_in(rows_apply_kernel<KT>, sm, granted);                              \
        launch(rows_apply_kernel<KT>, grid, 256, sm, st, o, n, k, G);                 \
    }
    KH_ROWS_SWITCH
#undef KH_ROWS_CALL
}

void rows_split(const float* Vw, const int* live, int n, int k, float* Vl, float* R, uint64_t seed, uint64_t stream,
                double* G, cudaStream_t st) {
    const int grid = (n + kRows - 1) / kRows;
#define KH_ROWS_CALL(KT) launch(rows_split_kernel<KT>, grid, 256, 0, st, Vw, live, n, k, Vl, R, seed, stream, G)
    KH_ROWS_SWITCH
#undef KH_ROWS_CALL
}

void rows_project(const float* Vl, const double* C, int n, int k, float* R, double* G, cudaStream_t st) {
    const int grid = (n + kRows - 1) / kRows;
#define KH_ROWS_CALL(KT)                                                              \
    {                                                                                 \
        constexpr size_t sm = sizeof(float) * 16 * KT * (2 * kRows + 16 * KT);        \
        static std::atomic<size_t> granted[kMaxDevices] = {};                         \
        smem_opt_in(rows_project_kernel<KT>, sm, granted);                            \
        launch(rows_project_kernel<KT>, grid, 256, sm, st, Vl, C, n, k, R, G);            \
    }
    KH_ROWS_SWITCH
#undef KH_ROWS_CALL
}

}  // namespace kh
