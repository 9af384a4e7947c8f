// tc_gemm.cuh -- a persistent tcgen05 GEMM with the boundary's epilogues fused in, for the
// shapes the fused boundary kernels do not take or are slower at (m = r = 128 and wider, m != r,
// the m = 64 encoder backward, few wide tokens: tc_preferred() in tc.cu):
// there the two linear layers of Sec. 3.2's encoder and decoder, and their gradients, become a
// chain of products C = A . B (bf16 operands, fp32 accumulation in TMEM), each with the
// element-wise step that follows it in the chain (phi, phi', the identity-path merge of Eq. Pid,
// the residual-gradient update) applied to the accumulator before it leaves the chip.
//
//   C[M x N] = sum over k of A[m][k] . B[k][n]
//   A: K-major (stored M x K row-major) or MN-major (stored K x M row-major, i.e. A^T in memory)
//   B: K-major (stored N x K row-major) or MN-major (stored K x N row-major)
//
// Work units are (row block, BN-column block, K split); unit u runs on CTA (pair) u mod grid
// (n fastest, then m, then the split: CTAs running at the same time share their A block and,
// across a wave, their B rows in L2). The row block is 256 rows on a pair of CTAs with two-CTA
// MMAs (PAIR: every product of more than 128 columns and 128 rows), else 128 rows on one CTA. Per
// CTA:
//   producer warp  : TMA loads of 64-deep K slices of A (128 x 64) and B (BN x 64; PAIR: half of
//                    it), 128-byte swizzle, into a ring of NST stages
//   MMA warp       : four 128 x BN x 16 (PAIR: 256 x BN x 16, issued by the even CTA) tcgen05.mma
//                    per stage into one of two TMEM accumulators (double-buffered: the next
//                    unit's products overlap this unit's epilogue)
//   With ALO the A operand is a bf16 pair hi + lo (hi = a value rounded to bf16, lo = the
//   rounded remainder, two matrices of the same shape): each stage holds both A tiles and the
//   MMA warp issues hi . B and lo . B into the same accumulator, so the product sees A to about
//   16 significant bits (used where the result crosses the boundary, B and dB, and for the
//   decoder's dWd2 = G^T . dY, a long sum over tokens whose terms cancel for real gradients).
//   epilogue warps : eight warps, two per TMEM lane quarter splitting the columns: TMEM ->
//                    registers (one output row per thread, 32 columns at a time) -> the
//                    epilogue's element-wise step -> shared-memory boxes -> TMA stores (TS), or
//                    straight to global memory
// What bounds it: long products (K = d or K = tokens) the tensor cores (d = 8192, m = 512: 533 to
// 582 cycles a 64-deep slice on pairs, 512 at their rate; the last round of units is uneven);
// products with K = m <= 512 that write T x d the epilogue and the stores (m = 512: dF 274 us with
// one thread's dX read-modify-write and 128-thread boxes, 190 us now, 537 MB and 275 GFLOP); N <= 128
// with K = d the reading of A.
// Out-of-range rows, columns and K are read as zeros by TMA and never written, so any M, N, K
// with 16-byte row pitches work. Each output element is summed by one CTA in K order (a split-K
// launch writes per-split fp32 slots that a second kernel adds in slot order), so results are
// bitwise reproducible.
#pragma once

#include "common.cuh"
#include "tc_common.cuh"

namespace resbm {
namespace tc {

// ---- CTA pairs (cta_group::2): the two CTAs of a cluster of 2 work on one 256-row tile -------------
// tma_load_2d whose bytes complete on an mbarrier of either CTA of the pair (`bar` from map_shared)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *m, int32_t x, int32_t y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// D (+)= A * B over both CTAs, issued by one thread of the even CTA: A's rows 0..127 and the first half
// of B's columns from its own shared memory, the rest from the odd CTA's (the same offsets); each CTA's
// TMEM receives its own 128 rows of D.
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                              bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}

// Arrive on the mbarrier at the same offset in the CTAs of `mask` (3: both, 1: the even one) when every
// pair MMA issued so far has completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar, uint16_t mask = 3)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"(mask)
        : "memory");
}

// tmem_alloc / tmem_dealloc of a pair: executed by one warp of each of the two CTAs
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// The element-wise step after the product (acc = the fp32 accumulator of one output element at
// row `row`, column `col`; phi and phi' as in common.cuh; every bf16 result rounded once to
// nearest even).
// `lo` (if set) receives the rounded remainder of the bf16 activation result named below, so that
// a later product can use it as a hi + lo pair.
enum GemmEpMode : int {
    GEP_F32 = 0,   // out f32 = acc (with split-K: slot ks at out + ks * split_stride)
    GEP_BF16,      // out bf16 = acc
    GEP_P_A,       // out f32 = acc (if out), out2 bf16 = phi(acc) (lo: its remainder)  (P, A)
    GEP_ADD_AUX,   // out bf16 = acc + aux[row][col] for col < aux_cols, acc elsewhere  (B, Y, dB)
    GEP_ACT,       // out bf16 = phi(acc) (lo: its remainder), out2 f32 = acc if out2   (G, Q)
    GEP_DACT,      // out bf16 = acc * phi'(aux f32) (lo: its remainder), out2 bf16 = phi(aux) if
                   // out2                                                              (dQ; dP, A)
    GEP_DF,        // out bf16 = acc; rmw[row][col] += aux[row][col] for col < aux_cols (dF; dX += dB)
    GEP_AXPBY,     // out bf16 = alpha * acc + beta * aux[row][col] (aux bf16; the Newton-Schulz steps)
};

struct GemmEp {
    int mode, act;
    void *out;           // ldo elements per row
    int64_t ldo;
    void *out2;          // ldo2 elements per row
    int64_t ldo2;
    const void *aux;     // bf16 (ADD_AUX, DF) or f32 (DACT); lda elements per row
    int64_t lda, aux_cols;
    __nv_bfloat16 *rmw;  // DF: ldr elements per row
    int64_t ldr;
    int64_t split_stride;
    __nv_bfloat16 *lo;   // P_A, ACT, DACT: the remainder of the bf16 activation result (same pitch)
    float alpha, beta;   // AXPBY
    // ENCP launches (the encoder fused into the FFN down-projection): F = acc rounded to bf16
    // (stored at out if set), and the partial P_slice = F_tile . We1[cols of the tile] summed over
    // half of the unit's columns, written to slot (nb * 2 + half) of pslots (slots T x pm fp32,
    // slot_stride apart)
    const __nv_bfloat16 *we1;   // d x pm
    float *pslots;
    int64_t slot_stride;
    int pm;
};

struct GemmShape {
    int64_t M, N, K;
    int64_t kc;          // K per split, a multiple of 64
    int nm, nn, splits;
    int64_t units;       // nm * nn * splits
    // Row-balanced launch (one column block, one split, more row blocks than CTAs): CTA b takes the rows
    // [b * rpc, (b + 1) * rpc), rpc a multiple of 32, in 128-row units and a last one of rpc % 128 rows; 0: off.
    // Such a product is bound by reading A, and with whole 128-row blocks some CTAs read one block more than
    // others (256 blocks on 152 SMs: 2 against 1; 224 rows each instead). What it reads at is the bytes in flight,
    // so these launches keep one store box a warp and 64-column tiles where N allows: 6 stages of 16 KB of A, or 8.
    int rpc;
    int bnv;             // columns per unit (BN; on pairs with an MN-major A a multiple of 32 up to BN)
    int turn;            // row blocks between shifts of the column blocks' order (gemm_unit)
    int pc;              // 64-deep K slices per piece of a sum (GemmCfg's HALVES and PIECES)
};

// Sums in pieces. The tensor core truncates as it adds to its accumulator, an error that grows with the number of
// MMAs in one accumulator. Where a chain replaces a fused kernel whose accumulators hold shorter sums, the unit's
// sum runs in pieces of GemmShape::pc slices, added in fp32 (to nearest) in K order.
// HALVES: the products of up to 64 columns over d (P, dQ): two accumulators a unit, added as the epilogue reads
// them. P over K = 8192, error against 64 bits: one accumulator 9.1e-6, the fused kernel 8.4e-6.
// PIECES: the weight gradients of hi + lo operands, whose sums over the tokens are long: pieces alternate between
// the two accumulators, and the epilogue warps add them in registers while the next piece runs. dWd2 at m = 64 over
// 8192 tokens a split: one accumulator 1.9e-5, the fused kernel 2.5e-6 (~300 tokens in one).
constexpr bool gemm_halves(int bn, bool amn, bool alo, bool encp, bool pair, bool bm2, int ts)
{
    return (bn == 64 || (bn == 128 && ts == 0)) && !amn && !alo && !encp && !pair && !bm2;   // (TS: N <= 64 by BN = 64)
}
constexpr bool gemm_pieces(bool amn, bool alo, bool pair, bool bm2) { return amn && alo && !pair && !bm2; }

// BM2: 256-row units, two 128-row A sub-tiles per stage against one B tile, the two halves'
// accumulators side by side in TMEM (one unit at a time: no accumulator double buffering).
// PAIR: CTA pairs (cta_group::2) on 256-row units: a stage of each CTA holds its own 128 rows of A and
// half of the B tile.
// TS: the outputs leave by TMA stores from shared-memory boxes, two 4 KB boxes per epilogue warp (one
// fills while the other's store reads it; RB: one box), each warp on its own: no barrier between warps. 1: one bf16
// output in boxes of 32 rows x 64 columns (128-byte swizzle); 2: an fp32 output in boxes of 32 rows x 32
// columns and / or up to two bf16 outputs of 32 x 32 in one box (64-byte rows; BN = 64 a third in the next box: dP's hi and lo
// and phi(P); the encoder backward at m = 64, T = 32768, d = 1024 65.5 us with dP by per-thread stores, 60.6 so). Per-thread 16-byte stores put 32 different rows
// in a warp instruction: they, not the products, set the pace where K is short.
// ENCP: one box of 32 rows x 64 columns per warp (F as the partial P's operand, and for F's store) and
// We1's rows of the unit's columns.
template <int BN_, bool ALO_ = false, bool BM2_ = false, int TS_ = 0, bool PAIR_ = false, bool ENCP_ = false, bool RB_ = false,
          bool HALVES_ = false>
struct GemmCfg {
    static constexpr int BN = BN_;
    static constexpr uint32_t A_TILE = 128 * 64 * 2;        // 128 rows x 64 K, bf16
    static constexpr uint32_t A_STAGE = A_TILE * (ALO_ ? 2 : 1) * (BM2_ ? 2 : 1);   // hi (+ lo), per half
    static constexpr uint32_t B_STAGE = (PAIR_ ? BN_ / 2 : BN_) * 64 * 2;   // BN (PAIR: BN / 2) rows x 64 K, bf16
    static constexpr uint32_t STAGE = A_STAGE + B_STAGE;
    static constexpr uint32_t BOX = 32 * 128;               // a staging box: 32 rows of 128 bytes
    static constexpr int NBOX = TS_ && !RB_ ? 2 : TS_ || ENCP_ ? 1 : 0;      // boxes per epilogue warp
    static constexpr uint32_t STG_WARP = NBOX * BOX;
    static constexpr uint32_t WE1_HALF = 128 * 64;          // ENCP: 128 columns' rows of We1 (up to 32 wide)
    static constexpr uint32_t STG_BYTES = 8 * STG_WARP + (ENCP_ ? 2 * WE1_HALF : 0);
    // stages: 4 at BN = 256, 6 at 128 (3, 4 with lo; 3 for BM2; PAIR: 6 and 8, 4 and 5 with lo); beside the
    // boxes of TS 3 at BN = 256 (2 with lo; PAIR: 5 and 3), from a larger share of the 227 KB
    static constexpr int NST = ((STG_BYTES ? 224 : 200) * 1024 - (int)STG_BYTES) / (int)STAGE;
    static constexpr uint32_t OFF_STG = NST * STAGE;        // 1024-aligned (STAGE is)
    static constexpr uint32_t OFF_WE1 = OFF_STG + 8 * STG_WARP;
    static constexpr uint32_t SMEM_BYTES = NST * STAGE + STG_BYTES + 1024;
    static_assert(SMEM_BYTES <= 232448 - 512, "shared memory budget");
    static constexpr uint32_t TMEM_COLS = (HALVES_ ? 4 : 2) * BN_;   // two accumulators (HALVES: two of two)
    static_assert(TMEM_COLS <= 512, "TMEM budget");
    static constexpr int EPI = 256;                         // epilogue threads (8 warps)
    static constexpr int THREADS = 64 + EPI;
};

// (in 32 bits, which hold every unit, as the host checks: a 64-bit division costs 0.2 us, and the first ones delay
// the first load)
__device__ __forceinline__ void gemm_unit(const GemmShape &g, uint32_t u, int &mb, int &nb, int &ks)
{
    const uint32_t nn = (uint32_t)g.nn, rest = u / nn;
    // The column blocks that carry the identity path's extra work must not keep falling to the same CTAs. With one
    // order of the columns, block 0 of row block t is unit t * nn, on worker t * nn mod W: only every gcd(nn, W)-th
    // worker, in turns of W / gcd row blocks. So each turn starts one column later: every worker in W row blocks
    // gets one. (A start that moves with every row block met the grid's stride instead: 16 x 20 blocks on 76 pairs
    // put four of the 16 identity blocks on one pair, T = 4096, d = 5120, r = 96 20.4 us; so 17.0.)
    const uint32_t at = u - rest * nn, shift = rest < (uint32_t)g.turn ? 0 : rest / (uint32_t)g.turn % nn;
    nb = (int)(at >= shift ? at - shift : at + nn - shift);
    ks = g.splits > 1 ? (int)(rest / (uint32_t)g.nm) : 0;
    mb = (int)rest - ks * g.nm;
}

// ---- the epilogue's element-wise steps on 32 consecutive columns of one row ----------------
__device__ __forceinline__ void st_bf16x32(__nv_bfloat16 *dst, const float (&v)[32], int nv)
{
    if (nv == 32) {
        uint4 *o = reinterpret_cast<uint4 *>(dst);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                __nv_bfloat162 h = __floats2bfloat162_rn(v[8 * q + 2 * e], v[8 * q + 2 * e + 1]);
                pk[e] = *reinterpret_cast<uint32_t *>(&h);
            }
            o[q] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
    } else {   // every index a constant (no dynamic indexing of the register array)
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < nv) dst[j] = __float2bfloat16_rn(v[j]);
    }
}

// hi = v rounded to bf16 at dst, lo = (v - hi) rounded to bf16 at dst_lo (if set)
__device__ __forceinline__ void st_bf16x32_split(__nv_bfloat16 *dst, __nv_bfloat16 *dst_lo, float (&v)[32], int nv)
{
    st_bf16x32(dst, v, nv);
    if (dst_lo) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] -= __bfloat162float(__float2bfloat16_rn(v[j]));
        st_bf16x32(dst_lo, v, nv);
    }
}

__device__ __forceinline__ void st_f32x32(float *dst, const float (&v)[32], int nv)
{
    if (nv == 32) {
        float4 *o = reinterpret_cast<float4 *>(dst);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < nv) dst[j] = v[j];
    }
}

__device__ __forceinline__ void st_f32x16(float *dst, const float (&v)[16], int nv)
{
    if (nv == 16) {
        float4 *o = reinterpret_cast<float4 *>(dst);
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < nv) dst[j] = v[j];
    }
}

__device__ __forceinline__ void ld_bf16x32(const __nv_bfloat16 *src, float (&x)[32], int nv)
{
    if (nv == 32) {
        load_bf16_row<32>(src, x);
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = j < nv ? __bfloat162float(src[j]) : 0.0f;
    }
}

__device__ __forceinline__ void ld_f32x32(const float *src, float (&x)[32], int nv)
{
    if (nv == 32) {
        const float4 *s = reinterpret_cast<const float4 *>(src);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 t = s[q];
            x[4 * q] = t.x; x[4 * q + 1] = t.y; x[4 * q + 2] = t.z; x[4 * q + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = j < nv ? src[j] : 0.0f;
    }
}

// v: the accumulator's columns [col, col + nv) of row `row` (nv <= 32; the vector forms need
// nv == 32 and 16-byte aligned rows, which the host guarantees for nv == 32)
__device__ __forceinline__ void gemm_epilogue(const GemmEp &ep, int64_t row, int64_t col, float (&v)[32], int nv,
                                              int ks)
{
    switch (ep.mode) {
    case GEP_F32:
        st_f32x32(static_cast<float *>(ep.out) + ks * ep.split_stride + row * ep.ldo + col, v, nv);
        break;
    case GEP_BF16:
        st_bf16x32(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col, v, nv);
        break;
    case GEP_P_A:
        if (ep.out) st_f32x32(static_cast<float *>(ep.out) + row * ep.ldo + col, v, nv);
        act_fast_row<32>(ep.act, v);
        st_bf16x32_split(static_cast<__nv_bfloat16 *>(ep.out2) + row * ep.ldo2 + col,
                         ep.lo ? ep.lo + row * ep.ldo2 + col : nullptr, v, nv);
        break;
    case GEP_ADD_AUX:
        if (col < ep.aux_cols) {
            const int na = ep.aux_cols - col < nv ? (int)(ep.aux_cols - col) : nv;
            float x[32];
            ld_bf16x32(static_cast<const __nv_bfloat16 *>(ep.aux) + row * ep.lda + col, x, na);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = j < na ? v[j] + x[j] : v[j];
        }
        st_bf16x32(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col, v, nv);
        break;
    case GEP_ACT:
        if (ep.out2) st_f32x32(static_cast<float *>(ep.out2) + row * ep.ldo2 + col, v, nv);
        act_fast_row<32>(ep.act, v);
        st_bf16x32_split(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col,
                         ep.lo ? ep.lo + row * ep.ldo + col : nullptr, v, nv);
        break;
    case GEP_DACT: {
        float x[32], dx[32];
        ld_f32x32(static_cast<const float *>(ep.aux) + row * ep.lda + col, x, nv);
        dact_fast_row<32>(ep.act, x, dx);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] *= dx[j];
        st_bf16x32_split(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col,
                         ep.lo ? ep.lo + row * ep.ldo + col : nullptr, v, nv);
        if (ep.out2) {
            act_fast_row<32>(ep.act, x);
            st_bf16x32(static_cast<__nv_bfloat16 *>(ep.out2) + row * ep.ldo2 + col, x, nv);
        }
        break;
    }
    case GEP_AXPBY: {
        float x[32];
        ld_bf16x32(static_cast<const __nv_bfloat16 *>(ep.aux) + row * ep.lda + col, x, nv);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = fmaf(ep.alpha, v[j], ep.beta * x[j]);
        st_bf16x32(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col, v, nv);
        break;
    }
    case GEP_DF:
        st_bf16x32(static_cast<__nv_bfloat16 *>(ep.out) + row * ep.ldo + col, v, nv);
        if (ep.rmw && col < ep.aux_cols) {
            const int na = ep.aux_cols - col < nv ? (int)(ep.aux_cols - col) : nv;
            float x[32], y[32];
            __nv_bfloat16 *r = ep.rmw + row * ep.ldr + col;
            ld_bf16x32(r, y, na);
            ld_bf16x32(static_cast<const __nv_bfloat16 *>(ep.aux) + row * ep.lda + col, x, na);
#pragma unroll
            for (int j = 0; j < 32; ++j) y[j] += x[j];
            st_bf16x32(r, y, na);
        }
        break;
    }
}

// rmw[row][col] += aux[row][col] (bf16, added in fp32) for the 32 rows from row0 (rows < M) and the columns
// [col0, col1), one warp, in whole 128-byte row pieces (eight lanes a row). One row per thread between the
// accumulator and the store this cost 9000 cycles a box of 64 columns. (16 rows at a time: 32 made the
// epilogue loop spill.)
__device__ __forceinline__ void rmw_rows(const GemmEp &ep, int64_t row0, int64_t M, int64_t col0, int64_t col1)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (; col0 < col1; col0 += 64) {
        const int64_t col = col0 + 8 * (lane & 7);
        if (col >= col1) continue;
#pragma unroll 1
        for (int64_t row = row0 + (lane >> 3); row < row0 + 32; row += 16) {
            uint4 x[4], y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (row + 4 * i < M) {
                    x[i] = __ldg(reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(ep.aux) + (row + 4 * i) * ep.lda + col));
                    y[i] = *reinterpret_cast<const uint4 *>(ep.rmw + (row + 4 * i) * ep.ldr + col);
                }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (row + 4 * i < M)
                    *reinterpret_cast<uint4 *>(ep.rmw + (row + 4 * i) * ep.ldr + col) =
                        make_uint4(add_bf16x2(y[i].x, x[i].x), add_bf16x2(y[i].y, x[i].y), add_bf16x2(y[i].z, x[i].z),
                                   add_bf16x2(y[i].w, x[i].w));
        }
    }
}

// tma_lo: the lo matrix of A (same shape and layout as A; read only with ALO; RB: A in boxes of the last
// unit's rows); tmo, tmo2, tmol: the
// outputs ep.out, ep.out2 and ep.lo in the boxes of the TS form (read only with TS; ENCP: tmo, if ep.out)
// ENCP: the epilogue of the encoder fused into the FFN down-projection (the GemmEp ENCP fields)
// instead of gemm_epilogue.
// BM2 (GemmCfg): units of 256 rows (two 128-row MMAs per K step sharing the B tile, ~128 flop per
// shared-memory byte against ~85), for long K where a unit's epilogue is short next to its
// products; not with ALO or PAIR.
// PAIR: CTA pairs (clusters of 2) run 256-row units with two-CTA MMAs (cta_group::2, 256 x BN x 16): CTA
// `rank` loads the rows 128 * rank .. + 127 of A and half of the B tile, all bytes counted on the even
// CTA's `full` barrier; the even CTA's MMA thread issues for both, and its commits free the stage and
// publish the accumulators in both (multicast). Each SM reads 96 operand rows a K step for 128 x 256
// products instead of 384 / 2, and 32 KB instead of 48 KB a stage keep six in flight.
// (For K-major B the tensor map's box is BN / 2 rows.)
// RB: row-balanced units (GemmShape::rpc).
template <int BN, bool AMN, bool BMN, bool ALO, bool ENCP = false, bool PAIR = false, bool BM2 = false,
          int TS = 0, bool RB = false>
__global__ void __launch_bounds__(320, 1)
    k_gemm(const __grid_constant__ CUtensorMap tma, const __grid_constant__ CUtensorMap tma_lo,
           const __grid_constant__ CUtensorMap tmb, const __grid_constant__ CUtensorMap tmo,
           const __grid_constant__ CUtensorMap tmo2, const __grid_constant__ CUtensorMap tmol, const GemmShape g,
           const GemmEp ep)
{
    constexpr bool HALVES = gemm_halves(BN, AMN, ALO, ENCP, PAIR, BM2, TS), PIECES = gemm_pieces(AMN, ALO, PAIR, BM2);
    using C = GemmCfg<BN, ALO, BM2, TS, PAIR, ENCP, RB, HALVES>;
    // (a compile-time property so that the other launches keep their index arithmetic)
    constexpr bool ROWS = RB;
    const int bnv = PAIR && AMN ? g.bnv : BN;
    static_assert(!RB || (BN <= 128 && !AMN && !ALO && !ENCP && !PAIR && !BM2 && TS), "row-balanced: K-major A, one column block");
    static_assert(!(BM2 && (ALO || PAIR)), "256-row units without hi + lo A or pairs");
    static_assert(!(TS && (ENCP || BM2)), "TMA-store epilogue: plain 128-row units or pairs");
    static_assert(!PIECES || (BMN && TS == 0 && !ENCP), "sums in pieces: the weight gradients on single CTAs");
    constexpr int MH = BM2 ? 2 : 1;   // 128-row halves per unit (g.nm counts units of 128 * MH rows)
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[C::NST], empty[C::NST], acc_full[2], acc_empty[2], done_bar;
    __shared__ uint32_t tmem_base_sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    auto k_steps = [&](int ks, int64_t &k0) -> int {
        k0 = (int64_t)ks * g.kc;
        int64_t k1 = k0 + g.kc;
        if (k1 > g.K) k1 = g.K;
        return (int)((k1 - k0 + 63) / 64);
    };
    // this CTA's units: every gridDim.x-th from blockIdx.x, or for a pair every (gridDim.x / 2)-th
    // pair unit from the cluster index, the row block 2 * (pair row block) + rank
    const uint32_t crank = PAIR ? cluster_rank() : 0u;
    const uint32_t u_first = PAIR ? cluster_index() : ROWS ? 0u : blockIdx.x;
    const uint32_t u_step = PAIR ? gridDim.x / 2 : ROWS ? 1u : gridDim.x;
    GemmShape gp = g;
    if (ROWS) gp.units = (g.rpc + 127) / 128;
    if (PAIR) {
        gp.nm = (g.nm + 1) / 2;
        gp.units = (int64_t)gp.nm * gp.nn * gp.splits;
    }
    const uint32_t units = (uint32_t)gp.units;
    auto unit_of = [&](uint32_t u, int &mb, int &nb, int &ks) {
        if (ROWS) {
            mb = (int)u;
            nb = ks = 0;
            return;
        }
        gemm_unit(gp, u, mb, nb, ks);
        if (PAIR) mb = 2 * mb + (int)crank;   // past the last row block: loads read zeros, nothing is stored
    };
    // first row of a unit, and the end of the rows this CTA may store
    auto row_of = [&](int mb) { return (ROWS ? (int64_t)blockIdx.x * g.rpc : (int64_t)0) + (int64_t)mb * 128; };
    const int64_t m_end = ROWS && (int64_t)(blockIdx.x + 1) * g.rpc < g.M ? (int64_t)(blockIdx.x + 1) * g.rpc : g.M;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::NST; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&acc_full[i]), 1);
            mbar_init(smem_u32(&acc_empty[i]), PAIR ? 2 * C::EPI / 32 : C::EPI);   // PAIR: both CTAs' warps, on the even CTA
        }
        mbar_init(smem_u32(&done_bar), 1);
        fence_mbar_init();
    }
    if (warp == 1) {
        if (PAIR) tmem_alloc_pair(smem_u32(&tmem_base_sh), C::TMEM_COLS);
        else tmem_alloc(smem_u32(&tmem_base_sh), C::TMEM_COLS);
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();   // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    // Barriers, TMEM and the pair were set up before the wait for the previous kernel, whose last
    // CTAs may still run: only what follows touches global memory.
    griddep_wait();               // the previous kernel of the stream has completed
    griddep_launch_dependents();  // the next one may be scheduled on SMs as they free up
    const uint32_t tmem = tmem_base_sh;

    if (warp == 0) {
        // ---------------- producer ----------------
        if (elect_one()) {
            tma_prefetch_desc(&tma);
            if (ALO || ROWS) tma_prefetch_desc(&tma_lo);
            tma_prefetch_desc(&tmb);
            uint32_t it = 0;
            bool ok = true;
            for (uint32_t u = u_first; u < units && ok; u += u_step) {
                int mb, nb, ks;
                unit_of(u, mb, nb, ks);
                int64_t k0;
                const int nk = k_steps(ks, k0);
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const uint32_t s = it % C::NST, ph = (it / C::NST) & 1;
                    if (!mbar_wait(smem_u32(&empty[s]), ph ^ 1)) {
                        ok = false;
                        break;
                    }
                    uint32_t bar = smem_u32(&full[s]);
                    const bool rest = ROWS && (mb + 1) * 128 > g.rpc;   // the shorter last unit: its own box (tma_lo)
                    if (!PAIR) {
                        mbar_expect_tx(bar, rest ? (uint32_t)(g.rpc % 128) * 128u + C::B_STAGE : C::STAGE);
                    } else {   // both CTAs' bytes on the even CTA's barrier
                        if (crank == 0) mbar_expect_tx(bar, 2 * C::STAGE);
                        bar = map_shared(bar, 0);
                    }
                    auto load = [&](uint32_t dst, const CUtensorMap *m, int32_t x, int32_t y) {
                        if (PAIR) tma_load_2d_pair(dst, m, x, y, bar);
                        else tma_load_2d(dst, m, x, y, bar);
                    };
                    const uint32_t adst = smem_u32(smem + s * C::STAGE), bdst = adst + C::A_STAGE;
                    const int32_t kx = (int32_t)(k0 + 64 * kb);
                    if (BM2) {   // the unit's two 128-row A sub-tiles
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int32_t y = mb * 256 + 128 * h;
                            if (!AMN) {
                                tma_load_2d(adst + h * C::A_TILE, &tma, kx, y, bar);
                            } else {
                                tma_load_2d(adst + h * C::A_TILE, &tma, y, kx, bar);
                                tma_load_2d(adst + h * C::A_TILE + 8192, &tma, y + 64, kx, bar);
                            }
                        }
                    } else if (!AMN) {
                        load(adst, rest ? &tma_lo : &tma, kx, (int32_t)row_of(mb));
                        if (ALO) load(adst + C::A_TILE, &tma_lo, kx, mb * 128);
                    } else {
                        load(adst, &tma, mb * 128, kx);
                        load(adst + 8192, &tma, mb * 128 + 64, kx);
                        if (ALO) {
                            load(adst + C::A_TILE, &tma_lo, mb * 128, kx);
                            load(adst + C::A_TILE + 8192, &tma_lo, mb * 128 + 64, kx);
                        }
                    }
                    if (PAIR) {   // this CTA's half of B
                        // (a narrower unit's half ends inside the tile: what lies past it is loaded and not read)
                        if (!BMN) {
                            load(bdst, &tmb, kx, nb * bnv + (int)crank * (bnv / 2));
                        } else {
#pragma unroll
                            for (int j = 0; j < BN / 128; ++j)
                                load(bdst + j * 8192, &tmb, nb * bnv + (int)crank * (bnv / 2) + 64 * j, kx);
                        }
                    } else if (!BMN) {
                        tma_load_2d(bdst, &tmb, kx, nb * BN, bar);
                    } else {
#pragma unroll
                        for (int j = 0; j < BN / 64; ++j) tma_load_2d(bdst + j * 8192, &tmb, nb * BN + 64 * j, kx, bar);
                    }
                }
            }
            // drain the loads still in flight before the CTA may exit; a pair's CTAs wait for the MMAs
            // that read them (whose commits arrive on both CTAs' stage barriers)
            const uint32_t n = it < (uint32_t)C::NST ? it : (uint32_t)C::NST;
            for (uint32_t k = 0; k < n; ++k) {
                const uint32_t j = it - 1 - k;
                if (!PAIR) mbar_wait(smem_u32(&full[j % C::NST]), (j / C::NST) & 1);
                else if (ok) mbar_wait(smem_u32(&empty[j % C::NST]), (j / C::NST) & 1);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if ((!PAIR || crank == 0) && elect_one()) {   // a pair's even CTA issues for both
            const uint32_t idesc = idesc_bf16(PAIR ? 256 : 128, (uint32_t)bnv, AMN, BMN);
            // stage-0 descriptors, advanced by (byte offset >> 4) in the start-address field.
            // K-major: rows of 128 bytes (64 K), 8-row groups 1024 bytes apart, a K step of 16 =
            // 32 bytes. MN-major: 64-wide blocks of 64 K rows (8 KB) 8192 bytes apart along M/N,
            // 8-row groups along K 1024 bytes apart, a K step of 16 = 16 rows = 2048 bytes.
            const uint32_t a0 = smem_u32(smem), b0 = a0 + C::A_STAGE;
            const uint64_t ad0 = AMN ? smem_desc(a0, 8192, 1024, kSwz128) : smem_desc(a0, 16, 1024, kSwz128);
            const uint64_t bd0 = BMN ? smem_desc(b0, 8192, 1024, kSwz128) : smem_desc(b0, 16, 1024, kSwz128);
            constexpr uint64_t AK = AMN ? (2048 >> 4) : (32 >> 4);
            constexpr uint64_t BK = BMN ? (2048 >> 4) : (32 >> 4);
            uint32_t it = 0, ti = 0;
            bool ok = true;
            for (uint32_t u = u_first; u < units && ok; u += u_step) {
                int mb, nb, ks;
                unit_of(u, mb, nb, ks);
                int64_t k0;
                const int nk = k_steps(ks, k0);
                const int pc = HALVES || PIECES ? g.pc : nk;
                for (int kp = 0; kp < nk && ok; kp += pc) {   // (one piece but for HALVES and PIECES)
                    // double-buffered accumulators; BM2: one pair of half accumulators, every unit
                    const uint32_t ab = BM2 ? 0u : (ti & 1);
                    if (!HALVES || kp == 0) {
                        const uint32_t eph = BM2 ? ((ti & 1) ^ 1) : (((ti >> 1) & 1) ^ 1);
                        ok = mbar_wait(smem_u32(&acc_empty[ab]), eph);
                        tc_fence_after();
                        if (!ok) break;
                    }
                    const uint32_t d_tmem = tmem + (HALVES ? (2 * ab + (kp ? 1 : 0)) * BN : ab * BN);
                    const int ke = nk - kp < pc ? nk : kp + pc;
                    for (int kb = kp; kb < ke; ++kb, ++it) {
                        const uint32_t s = it % C::NST, ph = (it / C::NST) & 1;
                        ok = mbar_wait(smem_u32(&full[s]), ph);
                        tc_fence_after();
                        if (!ok) break;
                        const uint64_t so = (uint64_t)((s * C::STAGE) >> 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            if (PAIR) {
                                mma_bf16_pair(d_tmem, ad0 + so + kk * AK, bd0 + so + kk * BK, idesc, kb > kp || kk > 0);
                                if (ALO)
                                    mma_bf16_pair(d_tmem, ad0 + so + (C::A_TILE >> 4) + kk * AK, bd0 + so + kk * BK, idesc, true);
                                continue;
                            }
                            mma_bf16(d_tmem, ad0 + so + kk * AK, bd0 + so + kk * BK, idesc, kb > kp || kk > 0);
                            if (ALO) mma_bf16(d_tmem, ad0 + so + (C::A_TILE >> 4) + kk * AK, bd0 + so + kk * BK, idesc, true);
                            if (BM2)   // the second 128-row half into the next BN columns
                                mma_bf16(d_tmem + BN, ad0 + so + (C::A_TILE >> 4) + kk * AK, bd0 + so + kk * BK, idesc,
                                         kb > kp || kk > 0);
                        }
                        // the stage is free once these MMAs are done (a pair's: in both CTAs)
                        if (PAIR) mma_commit_pair(smem_u32(&empty[s]));
                        else mma_commit(smem_u32(&empty[s]));
                    }
                    if (!ok) break;
                    if (HALVES && ke < nk) continue;   // the second half follows
                    if (PAIR) mma_commit_pair(smem_u32(&acc_full[ab]));
                    else mma_commit(smem_u32(&acc_full[ab]));
                    ++ti;
                }
            }
            if (PAIR) mma_commit_pair(smem_u32(&done_bar), 1);
            else mma_commit(smem_u32(&done_bar));
            mbar_wait(smem_u32(&done_bar), 0);
        }
    } else {
        // ---------------- epilogue warps ----------------
        const int q = warp & 3;                 // TMEM lane quarter this warp may access
        const int half = (warp - 2) >> 2;       // which half of the BN columns
        const int rin = q * 32 + lane;          // row within the 128-row block
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        uint32_t ti = 0, stg_it = 0;   // units; staging boxes filled
        uint8_t *const boxes = smem + C::OFF_STG + (warp - 2) * C::STG_WARP;   // this warp's
        // the next box, once its previous store has read it
        auto next_box = [&]() -> uint8_t * {
            if (lane == 0) bulk_wait_read<(C::NBOX > 1 ? 1 : 0)>();
            __syncwarp();
            return C::NBOX > 1 ? boxes + (stg_it++ & 1) * C::BOX : boxes;
        };
        // the warp's writes to the box are complete: store it at (col, row0)
        auto store_box = [&](const CUtensorMap &m, const uint8_t *box, int64_t col, int64_t row0) {
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_2d(&m, (int32_t)col, (int32_t)row0, smem_u32(box));
                bulk_commit();
            }
        };
        // 32 values of this thread's row as bf16, to bytes [at, at + 64) of the box row (pitch bytes)
        auto put_bf16 = [&](uint8_t *box, const float (&v)[32], uint32_t at, uint32_t pitch) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t pk[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) pk[i] = pack_bf16(v[8 * e + 2 * i], v[8 * e + 2 * i + 1]);
                *reinterpret_cast<uint4 *>(box + swz_offset((uint32_t)lane, at + 16 * e, pitch)) =
                    make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        };
        auto release_acc = [&](uint32_t ab) {   // every read of the accumulator is complete: it may be overwritten
            tc_fence_before();
            if (PAIR) {
                // (the arrival orders the TMEM reads only; a cluster-scope release would wait for the warp's
                // stores, ~3000 cycles a unit)
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(map_shared(smem_u32(&acc_empty[ab]), 0));
            } else {
                mbar_arrive(smem_u32(&acc_empty[ab]));
            }
        };
        bool two = false;   // HALVES: the unit has a second half (a split product's last split can be too short for one)
        // 32 columns of the accumulator `ab` from column c (warp-collective): the loads, and their end (HALVES: w, the
        // second half's)
        auto acc_ld32 = [&](uint32_t ab, int c, float (&v)[32], float (&w)[32]) {
            const uint32_t t = tmem + lane_base + ab * (HALVES ? 2 * BN : BN) + c;
            tmem_ld32(t, v);
            if (HALVES && two) tmem_ld32(t + BN, w);
        };
        auto acc_ready = [&](float (&v)[32], float (&w)[32]) {
            tmem_ld_wait();
            tmem_regs_ready(v);
            if (HALVES && two) {
                tmem_regs_ready(w);
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] += w[j];
            }
        };
        bool ok = true;
        for (uint32_t u = u_first; u < units && ok; u += u_step, ti += PIECES ? 0 : 1) {
            int mb, nb, ks;
            unit_of(u, mb, nb, ks);
            const uint32_t ab = BM2 ? 0u : (ti & 1);
            if (HALVES) {
                int64_t k0;
                two = k_steps(ks, k0) > g.pc;
            }
            if (ENCP) {   // this half's rows of We1 (zeros past the last column), while the products run
                constexpr int HC = BN / 2;
                uint8_t *w = smem + C::OFF_WE1 + half * C::WE1_HALF;
                named_barrier(1 + half, 128);   // the previous unit's have been read
                const int per = ep.pm / 8;      // 16-byte pieces per row, rows 64 bytes apart
                for (int e = (int)threadIdx.x - 64 - 128 * half; e < HC * per; e += 128) {
                    const int c = e / per, x = e - c * per;
                    const int64_t col = (int64_t)nb * BN + half * HC + c;
                    const uint4 v = col < g.N ? __ldg(reinterpret_cast<const uint4 *>(ep.we1 + col * ep.pm) + x)
                                              : make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint4 *>(w + swz_offset((uint32_t)c, 16 * x, 64)) = v;
                }
                named_barrier(1 + half, 128);
            }
            const int64_t ts_row0 = row_of(mb) + q * 32, ts_col0 = (int64_t)nb * BN + half * (BN / 2);
            if (TS == 1 && ep.mode == GEP_DF && ep.rmw) {
                const int64_t end = ts_col0 + BN / 2 < ep.aux_cols ? ts_col0 + BN / 2 : ep.aux_cols;
                if (ts_col0 < end) rmw_rows(ep, ts_row0, m_end, ts_col0, end);   // dX[:, :r] += dB, while the products run
            }
            if (PIECES) {
                float sum[BN / 32][16];   // this thread's columns
#pragma unroll
                for (int i = 0; i < BN / 32; ++i)
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[i][j] = 0.0f;
                int64_t k0;
                const int nk = k_steps(ks, k0);
#pragma unroll 1
                for (int kp = 0; kp < nk; kp += g.pc, ++ti) {
                    const uint32_t pb = ti & 1;
                    ok = mbar_wait(smem_u32(&acc_full[pb]), (ti >> 1) & 1);
                    tc_fence_after();
                    if (!ok) break;
#pragma unroll
                    for (int i = 0; i < BN / 32; ++i) {   // (16 at a time: 32 made the loop spill)
                        float v[16];
                        tmem_ld16(tmem + lane_base + pb * BN + half * (BN / 2) + 16 * i, v);   // warp-collective
                        tmem_ld_wait();
                        tmem_regs_ready(v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) sum[i][j] += v[j];
                    }
                    release_acc(pb);
                }
                if (!ok) break;
                const int64_t row = (int64_t)mb * 128 + rin;   // (the epilogue step is GEP_F32)
                float *dst = static_cast<float *>(ep.out) + ks * ep.split_stride + row * ep.ldo;
#pragma unroll
                for (int i = 0; i < BN / 32; ++i) {
                    const int64_t col = (int64_t)nb * BN + half * (BN / 2) + 16 * i;
                    if (row >= g.M || col >= g.N) continue;
                    st_f32x16(dst + col, sum[i], g.N - col < 16 ? (int)(g.N - col) : 16);
                }
                continue;
            }
            ok = mbar_wait(smem_u32(&acc_full[ab]), BM2 ? (ti & 1) : ((ti >> 1) & 1));
            tc_fence_after();
            if (!ok) break;
            if (ENCP) {
                // F as the FFN's bf16 output, 64 columns at a time in the warp's box (stored from there if
                // asked), then its share of P = F . We1 by warp MMAs on the box (m16n8k16: the tile's 128
                // tokens x 16 or 32 columns of P are too narrow for the idle TMEM columns, of which there
                // are none). On CUDA cores, one row per thread with We1 by broadcast loads, this took
                // 37 us a unit against 23 us of products.
                float pacc[2][4][4];
#pragma unroll
                for (int i = 0; i < 32; ++i) pacc[i >> 4][(i >> 2) & 3][i & 3] = 0.0f;
                const int64_t row0 = (int64_t)mb * 128 + q * 32;
                const uint32_t box = smem_u32(boxes), wb = smem_u32(smem + C::OFF_WE1 + half * C::WE1_HALF);
                const int nt8 = ep.pm / 8;
#pragma unroll 1
                for (int c0 = 0; c0 < BN / 2; c0 += 64) {
                    const uint32_t acc_col = ab * BN + half * (BN / 2) + c0;
                    float v[2][32];
                    tmem_ld32(tmem + lane_base + acc_col, v[0]);   // warp-collective: every lane
                    tmem_ld32(tmem + lane_base + acc_col + 32, v[1]);
                    if (lane == 0) bulk_wait_read<0>();            // the box's previous store has read it
                    tmem_ld_wait();
                    tmem_regs_ready(v[0]);
                    tmem_regs_ready(v[1]);
                    if (c0 + 64 >= BN / 2) release_acc(ab);
                    __syncwarp();                                  // (and every lane its previous fragments)
                    put_bf16(boxes, v[0], 0, 128);
                    put_bf16(boxes, v[1], 64, 128);
                    const int64_t col = (int64_t)nb * BN + half * (BN / 2) + c0;
                    if (ep.out && row0 < g.M && col < g.N) store_box(tmo, boxes, col, row0);
                    else __syncwarp();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t af[2][4];
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
                            ldsm4(af[mt], box + swz_offset(16 * mt + (lane & 15), 32 * k + 16 * (lane >> 4), 128));
#pragma unroll
                        for (int n = 0; n < 4; n += 2) {
                            if (n >= nt8) break;
                            uint32_t bf[4];   // (for an odd count of 8-column tiles the last is read and not used)
                            ldsm4t(bf, wb + swz_offset(c0 + 16 * k + (lane & 15), 16 * n + 16 * (lane >> 4), 64));
#pragma unroll
                            for (int mt = 0; mt < 2; ++mt) {
                                mma16816(pacc[mt][n], af[mt], bf[0], bf[1]);
                                if (n + 1 < nt8) mma16816(pacc[mt][n + 1], af[mt], bf[2], bf[3]);
                            }
                        }
                    }
                }
                float *slot = ep.pslots + (int64_t)(nb * 2 + half) * ep.slot_stride;
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int64_t row = row0 + 16 * mt + 8 * h + (lane >> 2);
                        if (row >= g.M) continue;
#pragma unroll
                        for (int n = 0; n < 4; ++n)
                            if (n < nt8)
                                *reinterpret_cast<float2 *>(slot + row * ep.pm + 8 * n + 2 * (lane & 3)) =
                                    make_float2(pacc[mt][n][2 * h], pacc[mt][n][2 * h + 1]);
                    }
                continue;
            }
            if (TS) {
                const int64_t row0 = ts_row0, row = row0 + lane;
                constexpr int CW = TS == 1 ? 64 : 32;   // columns at a time
#pragma unroll 1
                for (int c0 = half * (BN / 2); c0 < (half + 1) * (BN / 2); c0 += CW) {
                    const int64_t col0 = (int64_t)nb * bnv + c0;
                    const bool last = c0 + CW >= (half + 1) * (BN / 2);
                    float v[CW / 32][32];
                    float w[32];   // (HALVES: the second half)
#pragma unroll
                    for (int h = 0; h < CW / 32; ++h) acc_ld32(ab, c0 + 32 * h, v[h], w);
                    if (row0 >= m_end || col0 >= g.N || c0 >= bnv) {   // nothing of it exists (the same for the whole warp)
                        tmem_ld_wait();
                        if (last) release_acc(ab);
                        continue;
                    }
                    if (TS == 1) {
                        uint8_t *box = next_box();
                        tmem_ld_wait();
#pragma unroll
                        for (int h = 0; h < CW / 32; ++h) tmem_regs_ready(v[h]);
                        if (last) release_acc(ab);
#pragma unroll
                        for (int h = 0; h < CW / 32; ++h) {
                            const int64_t col = col0 + 32 * h;
                            // the identity path's columns; AXPBY: every column
                            if ((ep.mode == GEP_ADD_AUX || ep.mode == GEP_AXPBY) && row < m_end && col < ep.aux_cols) {
                                const int na = ep.aux_cols - col < 32 ? (int)(ep.aux_cols - col) : 32;
                                float x[32];
                                ld_bf16x32(static_cast<const __nv_bfloat16 *>(ep.aux) + row * ep.lda + col, x, na);
                                if (ep.mode == GEP_AXPBY) {
#pragma unroll
                                    for (int j = 0; j < 32; ++j) v[h][j] = fmaf(ep.alpha, v[h][j], ep.beta * x[j]);
                                } else {
#pragma unroll
                                    for (int j = 0; j < 32; ++j) v[h][j] = j < na ? v[h][j] + x[j] : v[h][j];
                                }
                            }
                            put_bf16(box, v[h], 64 * h, 128);
                        }
                        store_box(tmo, box, col0, row0);
                    } else {
                        // x: the pre-activation (P, Q) the element-wise step works on
                        float x[32];
                        uint8_t *box = next_box();
                        if (ep.mode == GEP_DACT && row < m_end)
                            ld_f32x32(static_cast<const float *>(ep.aux) + row * ep.lda + col0, x, g.N - col0 < 32 ? (int)(g.N - col0) : 32);
                        acc_ready(v[0], w);
                        if (last) release_acc(ab);
                        float *f32 = static_cast<float *>(ep.mode == GEP_ACT ? ep.out2 : ep.mode == GEP_DACT ? nullptr : ep.out);
                        if (f32) {   // P, Q, or a plain fp32 output
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                *reinterpret_cast<float4 *>(box + swz_offset((uint32_t)lane, 16 * e, 128)) =
                                    make_float4(v[0][4 * e], v[0][4 * e + 1], v[0][4 * e + 2], v[0][4 * e + 3]);
                            store_box(ep.mode == GEP_ACT ? tmo2 : tmo, box, col0, row0 + (int64_t)ks * g.M);
                            if (ep.mode == GEP_F32) continue;
                            box = next_box();
                        }
                        if (ep.mode == GEP_DACT) {
                            float dx[32];
                            if (ep.out2) act_dact_fast_row<32>(ep.act, x, x, dx);   // (one exponential for both)
                            else dact_fast_row<32>(ep.act, x, dx);
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[0][j] *= dx[j];
                        } else {
                            act_fast_row<32>(ep.act, v[0]);
                        }
                        if (BN == 64 && ep.mode == GEP_DACT && ep.lo && ep.out2) {   // three results: A = phi(P) in a box of its own
                            put_bf16(box, x, 0, 64);
                            store_box(tmo2, box, col0, row0);
                            box = next_box();
                        }
                        // the bf16 result in the box's first half, its remainder or A = phi(P) in the second
                        put_bf16(box, v[0], 0, 64);
                        const CUtensorMap *second = nullptr;
                        if (ep.lo) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) x[j] = v[0][j] - __bfloat162float(__float2bfloat16_rn(v[0][j]));
                            second = &tmol;
                        } else if (ep.mode == GEP_DACT && ep.out2) {
                            second = &tmo2;
                        }
                        if (second) put_bf16(box + C::BOX / 2, x, 0, 64);
                        fence_async_smem();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(ep.mode == GEP_P_A ? &tmo2 : &tmo, (int32_t)col0, (int32_t)row0, smem_u32(box));
                            if (second) tma_store_2d(second, (int32_t)col0, (int32_t)row0, smem_u32(box + C::BOX / 2));
                            bulk_commit();
                        }
                    }
                }
                continue;
            }
#pragma unroll 1
            for (int h = 0; h < MH; ++h) {   // the unit's 128-row halves (one unless BM2)
                const int64_t row = (int64_t)mb * (128 * MH) + 128 * h + rin;
                const uint32_t acc = ab + (uint32_t)h;
#pragma unroll 1
                for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
                    float v[32], w[32];
                    acc_ld32(acc, c, v, w);
                    acc_ready(v, w);
                    const int64_t col = (int64_t)nb * bnv + c;
                    if (col < g.N && row < g.M && c < bnv)
                        gemm_epilogue(ep, row, col, v, g.N - col < 32 ? (int)(g.N - col) : 32, ks);
                }
                if (h == MH - 1) release_acc(ab);
            }
        }
    }
    if ((TS || ENCP) && warp >= 2 && lane == 0) bulk_wait<0>();   // this warp's stores are done
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();   // neither CTA of a pair leaves, or frees TMEM, while the other may still address it
    if (warp == 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem, C::TMEM_COLS);
        else tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// The encoder's end after the fused down-projection, one token row per warp: lane j < m sums
// column j of the row's nslots partial slots in slot order (fp32; the lanes read the slots'
// rows coalesced), saves P if asked, and takes A_j = phi(P_j); lane n < r then forms
// E_n = sum over j of A_j . We2[j][n] (the A_j from lane j by shuffles, j in order) and stores
// B = X[:, :r] + E rounded to bf16. m, r <= 32.
__global__ void __launch_bounds__(256) k_enc_finish(const float *__restrict__ pslots, int nslots, int64_t slot_stride,
                                                    int64_t T, int m, int r, int act, float *__restrict__ P,
                                                    const __nv_bfloat16 *__restrict__ We2,
                                                    const __nv_bfloat16 *__restrict__ X, int64_t ldx,
                                                    __nv_bfloat16 *__restrict__ B)
{
    griddep_wait();
    griddep_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t >= T) return;   // whole warps
    float p = 0.0f;
    if (lane < m) {
        const float *src = pslots + t * m + lane;
        int s = 0;
        for (; s + 8 <= nslots; s += 8) {   // eight loads in flight, added in slot order
            float x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = __ldcs(src + (s + u) * slot_stride);
#pragma unroll
            for (int u = 0; u < 8; ++u) p += x[u];
        }
        for (; s < nslots; ++s) p += src[s * slot_stride];
        if (P) P[t * m + lane] = p;
    }
    const float a = lane < m ? act_f(act, p) : 0.0f;
    float e = 0.0f;
    for (int j = 0; j < m; ++j) {
        const float aj = __shfl_sync(0xffffffffu, a, j);
        if (lane < r) e = fmaf(aj, __bfloat162float(We2[j * r + lane]), e);
    }
    if (lane < r) B[t * r + lane] = __float2bfloat16_rn(__bfloat162float(X[t * ldx + lane]) + e);
}

}  // namespace tc
}  // namespace resbm
