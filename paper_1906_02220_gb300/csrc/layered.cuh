// Layered two-layer site contraction on the tensor cores: the shapes and the
// operand images shared by the kernel (layered.cu) and by the image builder
// (bond.cu).
//
// For nb blocks b (the chi^2 environment index pairs of an enlarged corner or
// an edge) the contraction is
//   out[b][ok][ob] = sum_p sum_{ik,ib} TL[ik][p][ok] Y[b][ib][ik] TL[ib][p][ob]
// with ik, ib, ok, ob pairs of virtual legs (D^2 values each) and p the
// physical index.  It runs as two GEMMs per tile of rows (b, ib):
//   ket layer  Z[(b,ib)][(p,ok)]  = sum_ik Y[(b,ib)][ik] TL[ik][(p,ok)]
//   bra layer  out[(b,ok)][ob]   += sum_(ib,p) Z[(b,ok)][(ib,p)] TL[(ib,p)][ob]
// over chunks of pc physical indices.  Z never leaves the SM: the ket GEMM
// accumulates it in tensor memory, the worker warps move it through shared
// memory into the (b,ok)-row layout, and the bra GEMM reads it back from
// tensor memory as its A operand.  The D^2 x D^2 double-layer index is never
// formed.
#pragma once

namespace kh {
namespace lay {

__host__ __device__ constexpr int pad_to(int x, int m) { return (x + m - 1) / m * m; }

// Tile shapes for bond dimension D (D^2 = d2), 1 or 3 MMA passes, and the
// operand type: TF32 (4-byte elements, K = 8 per MMA) or BF16 (2-byte
// elements, K = 16 per MMA, one pass).  Both move 32 bytes of K per MMA, so the
// shared-memory K blocks (128 bytes: 32 TF32 or 64 BF16 values) and the
// descriptor steps are the same; a tensor-memory column holds one TF32 or two
// BF16 values of the Z operand.
struct Plan {
    int esz = 4, kstep = 8;                  // element bytes; K per MMA
    int d2 = 0, bt = 0, rows = 0;            // D^2; blocks b per tile; rows (b, ib) used of 128
    bool fixed = false;                      // the fixed order of D <= kFixedOrderD with 3 passes
    int pc = 0, nb1 = 0, na2 = 0;            // physical indices per chunk; ket buffers; Z buffers
    int nacc1 = 1;                           // accumulators of a ket buffer
    int nm = 0, nacc2 = 0;                   // bra accumulators: of the leading products, and in all
    int n1 = 0, n1p = 0, k1p = 0, kb1 = 0;   // ket GEMM: N = pc D^2 (padded to 16), K = D^2 (padded to kstep)
    int n2p = 0, k2 = 0, k2p = 0, kb2 = 0;   // bra GEMM: N = D^2 (padded to 16), K = pc D^2 (padded to kstep)
    int zs = 0;                              // row stride (floats) of the shared-memory transpose buffer
    bool zswz = false;                       // its 16-byte chunks permuted by the row
    int acc1_cols = 0, out_cols = 0;         // columns of one ket / bra accumulator (32-aligned)
    int c_acc1 = 0, c_out = 0, c_a2 = 0, a2_cols = 0, c_y = 0, y_cols = 0, tmem = 0;   // tensor-memory columns
    int b1_bytes = 0, b2_bytes = 0;          // one (hi or lo) operand image
};

// Tensor-memory regions (512 columns): nb1 ket accumulators and nacc2 bra
// accumulators (32-column aligned), then the A operands, packed: na2 Z buffers
// and the Y tile, hi and lo with 3 passes.  The bra accumulators live through
// all chunks of a tile, and the tensor core truncates an accumulator at every
// instruction: with 3 passes the products of remainders have one of their own,
// so that they do not truncate the leading sum, which is spread over nm.  The
// plan picks pc (a power of two <= 16), nm, nb1 and na2, minimising a model of the
// tensor pipe: an MMA of N columns takes about 20 + 0.64 N clocks (measured on
// this kernel at N = 48 and 64 and on gemm3x.cu at 160), a chunk 100 more for
// its hand-off and 100 for each operand that has one buffer only.  Shared-memory
// operands use the 128-byte-swizzle K-major layout in K blocks of 128 bytes.
//
// With 3 passes and D <= kFixedOrderD the order and rounding of every sum are fixed
// (see make_dims in ctm.cu): operand heads are cut off and not rounded, the MMAs
// of a GEMM go pass by pass (hi hi, hi lo, lo hi) round-robin to four bra
// accumulators and to two ket accumulators a buffer (one at D = 3), summed in
// their order when read, and pc is the largest that fits.
constexpr int kFixedOrderD = 5;
__host__ __device__ constexpr Plan make_plan(int D, int npass, bool bf16 = false) {
    Plan P{};
    P.esz = bf16 ? 2 : 4;
    P.kstep = bf16 ? 16 : 8;
    const int per_block = 128 / P.esz;                  // K values per 128-byte block
    P.d2 = D * D;
    P.bt = P.d2 > 0 ? 128 / P.d2 : 0;
    P.rows = P.bt * P.d2;
    P.k1p = pad_to(P.d2, P.kstep);
    P.kb1 = (P.k1p + per_block - 1) / per_block;
    P.n2p = pad_to(P.d2, 16);
    if (P.bt < 1 || (bf16 && npass != 1)) return P;
    const int npl = npass == 3 ? 2 : 1;
    P.fixed = npass == 3 && D <= kFixedOrderD;
    double best = 1e30;
    for (int pc = 16; pc >= 1; pc /= 2) {
        const int n1p = pad_to(pc * P.d2, 16);
        if (n1p > (npass == 3 ? 96 : 128)) continue;    // a row of Z, or its two parts, fits the workers' registers
        const int k2p = pad_to(pc * P.d2, P.kstep);
        const int zcols = k2p * P.esz / 4, ycols = P.k1p * P.esz / 4;   // columns of one Z / Y operand
        const int nc = (16 + pc - 1) / pc;              // chunks at p = 16
        const int mm1 = (P.k1p / P.kstep) * npass, mm2 = (k2p / P.kstep) * npass;
        const double c1 = 20.0 + 0.64 * n1p, c2 = 20.0 + 0.64 * P.n2p;
        if (P.fixed && P.pc > 0) break;
        const int nacc1 = P.fixed && D != 3 ? 2 : 1;
        for (int nm = 2; nm >= 1; --nm)
            for (int nb = 4; nb >= 1; --nb) {
                const int nb1 = nb >= 3 ? 2 : 1, na2 = nb % 2 == 0 ? 2 : 1;
                const int nacc2 = P.fixed ? 4 : nm + (npass == 3 ? 1 : 0);
                if (nm > k2p / P.kstep) continue;
                const int cols = nb1 * nacc1 * pad_to(n1p, 32) + nacc2 * pad_to(P.n2p, 32) + npl * (na2 * zcols + ycols);
                if (cols > 512) continue;
                const double cost = nc * (mm1 * c1 + mm2 * c2 + 500.0 - 100.0 * (nb1 + na2)) - nm;
                if (cost >= best) continue;
                best = cost;
                P.pc = pc;
                P.nb1 = nb1;
                P.na2 = na2;
                P.nacc1 = nacc1;
                P.nm = nm;
                P.nacc2 = nacc2;
                P.n1 = pc * P.d2;
                P.n1p = n1p;
                P.k2 = pc * P.d2;
                P.k2p = k2p;
                P.kb2 = (k2p + per_block - 1) / per_block;
                // an odd number of 16-byte chunks a row, or whole 128-byte rows
                // with their chunks permuted by the row: conflict-free row reads
                P.zs = pad_to(P.k2, 4);
                P.zswz = P.zs % 32 == 0;
                // (without the odd stride, two-way conflicts, where it would cost the rings a stage)
                const int rings = 2 * npl * (n1p * P.kb1 + P.n2p * P.kb2) * 128;
                if (!P.zswz && (P.zs / 4) % 2 == 0 && 1024 + 2 * 128 * (P.zs + 4) * 4 + rings <= 230400) P.zs += 4;
                P.acc1_cols = pad_to(n1p, 32);
                P.out_cols = pad_to(P.n2p, 32);
                P.c_acc1 = 0;
                P.c_out = nb1 * nacc1 * P.acc1_cols;
                P.c_a2 = P.c_out + nacc2 * P.out_cols;
                P.a2_cols = zcols;
                P.c_y = P.c_a2 + na2 * npl * zcols;
                P.y_cols = ycols;
                P.tmem = 32;
                while (P.tmem < cols) P.tmem *= 2;
                P.b1_bytes = n1p * P.kb1 * 128;
                P.b2_bytes = P.n2p * P.kb2 * 128;
            }
    }
    return P;
}

// Byte offset of element (row r, k) of esz bytes in a K-major operand of
// `rows` rows with 128-byte swizzle: K blocks of 128 bytes, each block rows x
// 128 bytes, the 16-byte chunks of row r permuted by r mod 8.
__host__ __device__ inline int swz_offset(int r, int k, int rows, int esz = 4) {
    const int byte = k * esz, kb = byte >> 7, kc = byte & 127;
    return kb * rows * 128 + r * 128 + ((((kc >> 4) ^ (r & 7)) << 4) | (kc & 15));
}

// Inverse of swz_offset for an esz-aligned offset o: (row, k).
__host__ __device__ inline void swz_position(int o, int rows, int& r, int& k, int esz = 4) {
    const int kb = o / (rows * 128), rem = o % (rows * 128);
    r = rem / 128;
    const int ch = (rem % 128) >> 4;
    k = (kb * 128 + (((ch ^ (r & 7)) << 4) | (rem & 15))) / esz;
}

// Chunks of pc physical indices covering p.
__host__ __device__ inline int n_chunks(const Plan& P, int p) { return (p + P.pc - 1) / P.pc; }

}  // namespace lay

// Image sizes (floats) of one (kind, frame) operand set for p physical
// indices: ket images of all chunks, then bra images (hi, lo per chunk with
// 3 passes).  Zero when D has no tensor-core plan.
long long layered_img1_floats(int D, int p, int npass, bool bf16 = false);
long long layered_img2_floats(int D, int p, int npass, bool bf16 = false);

// Operand images of all (kind, frame) pairs from the FP64 site tensor
// Tm[p][D^4] (legs l, u, r, d of frame 0): img1 holds 8 x per1 floats, img2
// 8 x per2 (per1, per2 at least layered_img1_floats / layered_img2_floats for
// p), layout [kind][frame][chunk][hi, lo].  With Tbra given, the bra images
// come from Tbra (same shape) and the ket images from Tm: the mixed double
// layer of an operator applied to the ket layer only.
void build_layered_images(const double* Tm, int p, int D, int npass, bool bf16, float* img1, float* img2,
                          long long per1, long long per2, cudaStream_t st, const double* Tbra = nullptr);

// out[b][ok][ob] (row-major, nb x D^2 x D^2) from Y[b][ib][ik] (row-major,
// nb x D^2 x D^2) and the operand images of one (kind, frame).  Tensor-core
// passes npass = 1 (TF32, or BF16 with bf16 set) or 3 (3xTF32).  Time-outs
// set bits of *err.
void site_layered_tc(const float* Y, long long nb, int D, int p, const float* img1, const float* img2, float* out,
                     int npass, bool bf16, int* err, cudaStream_t st);

}  // namespace kh
