// One-sided (Hestenes) Jacobi SVD of a small dense FP64 matrix on a cluster of
// eight CTAs; the arithmetic and the stopping rules are those of the one-CTA
// kernel in jacobi.cuh.
//
// What bounds it: a round's chain (sums, rotation, cluster barrier), ~2 us; on one
// SM the FP64 pipe, which issues a warp's instruction in some 32 clocks, is the
// bound (5 us a round of 32 pairs).  A round here has four pairs on each of eight
// SMs, one warp a pair and one warp a sub-partition.
//
// Columns stay in shared memory.  In the round-robin ordering (circle method,
// as round_robin_pair) the columns of the upper seats move down by one seat each
// round and those of the lower seats up by one, so a CTA, which holds npc
// neighbouring seats, passes on two columns a round: the warp that has such a
// column in registers writes it straight into the neighbour's shared memory.
// Each of the two streams has npc + 1 buffers in turn, one more than it has seats,
// so that an arriving column never lands on one still read; a cluster barrier
// ends the round.
//
// The rotation's angle is found in FP32 (its error only leaves a residual of
// 1e-7 of the inner product for the next sweep); the rotation (c, s) itself is
// orthogonal to FP64 rounding.  So is the cosine of the stopping test.  Over 432
// matrices (random, graded, of low rank, clustered; 17 to 112 columns) residual,
// orthogonality and singular values are those of the one-CTA kernel or better
// (geometric means 1.5e-15, 9e-15 against 12e-15, 3.5e-15 against 5.0e-15).  The three sums of a pair are reduced over the
// warp together (six FP64 additions a lane instead of fifteen).
//
// 64 x 64 (the dense projector at D = 2, chi = 16): 0.50 ms in 3.9 sweeps, in one
// CTA 2.05 ms in 8.1 (columns of rounding noise no longer count towards the
// stopping test there).
#include <cooperative_groups.h>

#include "engine.cuh"

namespace kh {

namespace {

namespace cg = cooperative_groups;

constexpr int kClusterCtas = 8;
constexpr int kSeatsMax = 7;               // pairs per CTA: 2 * 8 * 7 = 112 columns
constexpr int kColsMax = 2 * kClusterCtas * kSeatsMax;

// Rotation (c, s) of two columns with squared norms a, b and inner product g:
// the angle in FP32, the rotation orthogonal in FP64.
__device__ __forceinline__ void rotation_fp32_angle(double a, double b, double g, double& c, double& s) {
    const float zeta = __fdividef(d2f_flush(b - a), 2.f * d2f_flush(g));
    const float az = fabsf(zeta);
    float t = az > 1e15f ? __fdividef(0.5f, az) : __fdividef(1.f, az + sqrtf(fmaf(az, az, 1.f)));
    if (!(az <= 3e38f)) t = 0.f;           // g below the FP32 range against b - a: nothing to rotate
    t = copysignf(t, zeta);
    const float cf = rsqrtf(fmaf(t, t, 1.f));
    c = f2d(cf);
    s = f2d(cf * t);
    // c^2 + s^2 = 1 + d with d ~ 2^-22: (1 + d)^-1/2 = 1 - d/2 + 3 d^2/8 to 1e-20
    const double d = fma(c, c, fma(s, s, -1.0)), f = fma(d, fma(d, 0.375, -0.5), 1.0);
    c *= f;
    s *= f;
}

// Sums of a, b and g over the warp: after the first two steps a quarter of the
// lanes holds each of them, so the other three steps add one value a lane.
__device__ __forceinline__ void reduce_abg(double& a, double& b, double& g, int lane) {
    const unsigned full = 0xffffffffu;
    double ab = (lane & 16) ? b : a;
    ab += __shfl_xor_sync(full, (lane & 16) ? a : b, 16);
    g += __shfl_xor_sync(full, g, 16);
    double x = (lane & 8) ? g : ab;
    x += __shfl_xor_sync(full, (lane & 8) ? ab : g, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(full, x, o);
    a = __shfl_sync(full, x, 0);
    b = __shfl_sync(full, x, 16);
    g = __shfl_sync(full, x, 8);
}

// RR rows per lane (32 RR >= k).  npc seats (column pairs) per CTA, one warp each.
template <int RR>
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(32 * kSeatsMax)
svd_cluster_kernel(const double* __restrict__ Xin, int k, int npc, double* __restrict__ s_out,
                   double* __restrict__ L_out, double* __restrict__ Q_out, int max_sweeps, double tol, double cut,
                   int* sweep_count, int nrel) {
    pdl_start();
    extern __shared__ double bufs[];       // 2 (npc + 1) + 1 columns of (X, Q), 32 RR rows each
    __shared__ double s_cn[kColsMax];      // squared column norms, by column
    __shared__ unsigned char s_top[kColsMax];
    __shared__ float s_c2[kClusterCtas * kSeatsMax];
    __shared__ int s_rot[kClusterCtas * kSeatsMax];
    __shared__ double s_red[kSeatsMax];
    constexpr int LD = 32 * RR, COL = 2 * LD;
    cg::cluster_group cl = cg::this_cluster();
    const int cta = (int)cl.block_rank(), lane = threadIdx.x & 31, i = threadIdx.x >> 5;   // warp = local seat
    const int nt = blockDim.x, tid = threadIdx.x;
    const int h = kClusterCtas * npc, kp = 2 * h, m = kp - 1, nb = npc + 1;
    const int gi = cta * npc + i;          // seat
    double* fixed = bufs + 2 * nb * COL;   // column 0 (CTA 0)
    auto top = [&](double* base, int b) { return base + b * COL; };
    auto bot = [&](double* base, int b) { return base + (nb + b) * COL; };
    auto modn = [&](int x) { return ((x % nb) + nb) % nb; };
    auto remote = [&](int rank) { return cl.map_shared_rank(bufs, rank); };

    // exact power-of-two scaling: largest |entry| in [1, 2)
    double mx = 0.0;
    for (int e = tid; e < k * k; e += nt) mx = fmax(mx, fabs(Xin[e]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_red[i] = mx;
    __syncthreads();
    for (int w = 0; w < npc; ++w) mx = fmax(mx, s_red[w]);
    int ex = 0;
    if (mx > 0.0) frexp(mx, &ex);
    const double scale = mx > 0.0 ? ldexp(1.0, 1 - ex) : 1.0;

    auto fill = [&](double* col, int c) {
#pragma unroll
        for (int j = 0; j < RR; ++j) {
            const int r = lane + 32 * j;
            col[r] = (r < k && c < k) ? Xin[(long long)r * k + c] * scale : 0.0;
            col[LD + r] = (r == c && c < k) ? 1.0 : 0.0;
        }
    };
    // seats of round 0: (0, 1) at seat 0, (1 + gi, kp - gi) at the others
    if (gi == 0) fill(fixed, 0);
    else fill(bot(bufs, modn(i)), kp - gi);
    fill(top(bufs, modn(i)), 1 + gi);
    cl.sync();

    const double tol_eff = fmax(tol, 2.0 * k * 1.1e-16), tol2 = tol_eff * tol_eff;
    const float floor2 = (float)(1e6 * 1.1e-16 * 1.1e-16);
    float prev2 = 1e30f;
    if (nrel <= 0 || nrel > kp) nrel = kp;
    // squared norms of the seat's columns (of a round r = 0), to every CTA
    auto share_norms = [&](int rr) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double* col = q == 0 ? top(bufs, modn(rr + i)) : (gi == 0 ? fixed : bot(bufs, modn(i - rr)));
            const int c = q == 0 ? 1 + gi : (gi == 0 ? 0 : kp - gi);
            double a = 0.0;
#pragma unroll
            for (int j = 0; j < RR; ++j) a = fma(col[lane + 32 * j], col[lane + 32 * j], a);
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane < kClusterCtas) *cl.map_shared_rank(&s_cn[c], lane) = a;
        }
        cl.sync();
    };
    int rr = 0, sw = 0;
    for (; sw < max_sweeps; ++sw) {
        if (nrel < kp) {
            // columns among the nrel largest must converge; the other pairs are
            // still rotated but do not keep the sweep loop alive
            share_norms(rr);
            for (int c = tid; c < kp; c += nt) {
                int rank = 0;
                const double cc = s_cn[c];
                for (int j = 0; j < kp; ++j) rank += (s_cn[j] > cc) || (s_cn[j] == cc && j < c);
                s_top[c] = rank < nrel;
            }
        } else {
            for (int c = tid; c < kp; c += nt) s_top[c] = 1;
        }
        __syncthreads();
        float c2max = 0.f;
        int rot = 0;
        // buffers and columns of this round, stepped from round to round (a
        // remainder by a runtime divisor costs more than the round's FP64 sums)
        int it = modn(rr + i), ib = modn(i - rr), arrive_t = modn(rr + npc), arrive_b = modn(-rr - 1);
        int tc = 1 + gi % m, bc = gi == 0 ? 0 : 1 + (m - gi) % m;
        for (int r = 0; r < m; ++r, ++rr) {
            double* tcol = top(bufs, it);
            double* bcol = gi == 0 ? fixed : bot(bufs, ib);
            const bool tfirst = tc < bc;                     // the column with the lower number comes first
            double u[RR], v[RR], qu[RR], qv[RR];
            const double *uc = tfirst ? tcol : bcol, *vc = tfirst ? bcol : tcol;
            double a = 0.0, b = 0.0, g = 0.0;
#pragma unroll
            for (int j = 0; j < RR; ++j) {
                const int row = lane + 32 * j;
                u[j] = uc[row];
                v[j] = vc[row];
                qu[j] = uc[LD + row];
                qv[j] = vc[LD + row];
                a = fma(u[j], u[j], a);
                b = fma(v[j], v[j], b);
                g = fma(u[j], v[j], g);
            }
            reduce_abg(a, b, g, lane);
            const double ab = a * b, g2 = g * g;
            bool turned = false;
            if (g != 0.0 && ab > 0.0) {
                const bool rel = s_top[tc] | s_top[bc];
                if (rel) {
                    // the squared cosine, in FP32 (columns below 1e-18 of the largest entry do not count)
                    const float fa = d2f_flush(a), fb = d2f_flush(b);
                    if (fa > 1e-36f && fb > 1e-36f) {
                        const float cs = d2f_flush(g) * rsqrtf(fa) * rsqrtf(fb);
                        c2max = fmaxf(c2max, cs * cs);
                    }
                }
                if (g2 > tol2 * ab) {
                    double c, s;
                    rotation_fp32_angle(a, b, g, c, s);
#pragma unroll
                    for (int j = 0; j < RR; ++j) {
                        const double nu = c * u[j] - s * v[j], nv = s * u[j] + c * v[j];
                        const double mu = c * qu[j] - s * qv[j], mv = s * qu[j] + c * qv[j];
                        u[j] = nu;
                        v[j] = nv;
                        qu[j] = mu;
                        qv[j] = mv;
                    }
                    rot |= rel;
                    turned = true;
                }
            }
            // where the two columns sit in the next round
            double *tdst = tcol, *bdst = bcol;
            if (gi == 0) tdst = npc > 1 ? bot(bufs, ib) : bot(remote(1), arrive_b);     // ib = -rr: seat 1 next
            else if (i == 0) tdst = top(remote(cta - 1), arrive_t);
            if (gi != 0 && i == npc - 1)
                bdst = cta < kClusterCtas - 1 ? bot(remote(cta + 1), arrive_b) : top(bufs, arrive_t);
            double *ud = tfirst ? tdst : bdst, *vd = tfirst ? bdst : tdst;
            const bool wu = turned || ud != uc, wv = turned || vd != vc;
#pragma unroll
            for (int j = 0; j < RR; ++j) {
                const int row = lane + 32 * j;
                if (wu) {
                    ud[row] = u[j];
                    ud[LD + row] = qu[j];
                }
                if (wv) {
                    vd[row] = v[j];
                    vd[LD + row] = qv[j];
                }
            }
            if (++it == nb) it = 0;
            if (--ib < 0) ib = npc;
            if (++arrive_t == nb) arrive_t = 0;
            if (--arrive_b < 0) arrive_b = npc;
            if (++tc == kp) tc = 1;
            if (gi != 0 && ++bc == kp) bc = 1;
            cl.sync();
        }
        // largest squared cosine and rotation flag over the cluster, once per sweep
        if (lane < kClusterCtas) {
            *cl.map_shared_rank(&s_c2[gi], lane) = c2max;
            *cl.map_shared_rank(&s_rot[gi], lane) = rot;
        }
        cl.sync();
        float bmax = 0.f;
        int brot = 0;
        for (int w = 0; w < h; ++w) {
            bmax = fmaxf(bmax, s_c2[w]);
            brot |= s_rot[w];
        }
        if (brot == 0) break;
        if (bmax < (float)(0.1 * tol_eff)) break;                // quadratic convergence: nothing left to rotate
        if (bmax < floor2 && bmax > 0.0625f * prev2) break;      // stagnated at the floor
        prev2 = bmax;
    }
    if (sweep_count && cta == 0 && tid == 0) atomicAdd(sweep_count, sw + 1);
    share_norms(rr);
    double smax = 0.0;
    for (int c = 0; c < k; ++c) smax = fmax(smax, sqrt(s_cn[c]));
    const double rscale = 1.0 / scale;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const double* col = q == 0 ? top(bufs, modn(rr + i)) : (gi == 0 ? fixed : bot(bufs, modn(i - rr)));
        const int c = q == 0 ? 1 + gi : (gi == 0 ? 0 : kp - gi);
        if (c >= k) continue;
        const double cc = s_cn[c], sc = sqrt(cc);
        int rank = 0;
        for (int j = lane; j < k; j += 32) rank += (s_cn[j] > cc) || (s_cn[j] == cc && j < c);
        for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        const double inv = (smax > 0.0 && sc > cut * smax) ? 1.0 / sc : 0.0;
#pragma unroll
        for (int j = 0; j < RR; ++j) {
            const int r = lane + 32 * j;
            if (r < k) {
                L_out[(long long)r * k + rank] = col[r] * inv;
                Q_out[(long long)r * k + rank] = col[LD + r];
            }
        }
        if (lane == 0) s_out[rank] = sc * rscale;
    }
    cl.sync();                             // no CTA leaves while another may still write to it
}

template <int RR>
void launch_cluster(const double* X, int k, int npc, double* s, double* L, double* Q, int max_sweeps, double tol,
                    double cut, cudaStream_t st, int* sweep_count, int nrel) {
    const size_t sm = sizeof(double) * (2 * (npc + 1) + 1) * 2 * 32 * RR;     // at most 34 KB
    launch(svd_cluster_kernel<RR>, kClusterCtas, 32 * npc, sm, st, X, k, npc, s, L, Q, max_sweeps, tol, cut,
           sweep_count, nrel);
}

}  // namespace

void svd_jacobi_cluster(const double* X, int k, double* s, double* L, double* Q, int max_sweeps, double tol,
                        double cut, cudaStream_t st, int* sweep_count, int nrel) {
    const int npc = (k + 2 * kClusterCtas - 1) / (2 * kClusterCtas);
    if (npc < 1 || npc > kSeatsMax) fail(KH_EINVAL, "svd_jacobi_cluster: k beyond limit");
#define KH_SVDC(RR) launch_cluster<RR>(X, k, npc, s, L, Q, max_sweeps, tol, cut, st, sweep_count, nrel)
    if (k <= 32) KH_SVDC(1);
    else if (k <= 64) KH_SVDC(2);
    else if (k <= 96) KH_SVDC(3);
    else KH_SVDC(4);
#undef KH_SVDC
}

}  // namespace kh
