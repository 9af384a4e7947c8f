// narrow.cuh -- the portable path for narrow bottlenecks (m, r <= 32; fp32, odd widths or unaligned
// pointers): each op of the boundary in one or two launches of CUDA-core kernels, fp32 throughout.
//
//   k_narrow_in    a tile of 16 token rows: the long product Z . W (K = d) split over the block's
//                  warps, then everything of the op that needs only the tile's m- and r-wide rows
//                  (encode forward: P, phi(P), B; decode backward: Q, phi(Q), dG, dQ, dB)
//   k_narrow_out   a tile of 16 token rows x 256 columns: the m-wide rows (decode forward: Q, phi(Q);
//                  encode backward: dP, phi(P)), then their product with W (K = m)
//   k_narrow_wgrad both weight gradients of a backward op: clusters of eight CTAs split the tokens of
//                  64 columns and add their partial sums in rank order through shared memory, so no
//                  partial reaches memory and no second launch sums them
//
// What bounds it: at T = 512, d = 256, r = 2 the step moves 2 MB and every launch is latency. The
// chain of tiled products this replaces took 13 launches on 1 to 8 CTAs that walked K = d or K = T
// alone (the weight gradients up to 120 us each): 378 us. Four launches (narrow_step) on 32 to 96 CTAs,
// chained by programmatic dependent launch, take 16 us (narrow_ok() has more sizes). Sums run in a fixed order (a warp's
// part of K, the warps in order; a rank's tokens, the ranks in order): bitwise reproducible.
#pragma once

#include "common.cuh"

namespace resbm {
namespace {

constexpr int kNT = 16;        // tokens per tile
constexpr int kNThr = 256;     // threads per block
constexpr int kNW = 32;        // the widest m and r
constexpr int kNChunk = 512;   // columns of Z staged at a time (k_narrow_in)
constexpr int kNCl = 8;        // CTAs per cluster (k_narrow_wgrad)

// The wide kernels (generic.cu) take any m and r; these hold a row of each in one warp's width. A step's
// time, wide -> narrow, fp32: T = 512, d = 256, r = m = 2: 371 -> 16 us; T = 2048, d = 1024, r = m = 8:
// 892 -> 52 us, r = m = 32: 990 -> 131 us; T = 16384, d = 2048, r = m = 16: 2.15 -> 0.64 ms; T = 65536,
// d = 64, r = m = 32: 1.77 -> 0.95 ms; T = 32768, d = 4096, r = m = 32: 5.8 -> 4.0 ms. bf16 alike. Of the ops alone
// only the forward ones at r = m = 32 and d <= 64 over many tokens are the wide kernels' (T = 65536, d = 64 encoder
// forward 45 -> 50 us, decoder forward 33.5 -> 36.3); the step's outputs are the ops', so they stay on one path.
inline bool narrow_ok(const resbm_desc &d) { return d.m <= kNW && d.r <= kNW; }

// element (t, j) of a rows x cols tile at src (row pitch ld) -> dst[t * 33 + j], zeros past `rows`
template <typename E>
__device__ __forceinline__ void stage_rows(const E *src, int64_t ld, int rows, int cols, float *dst)
{
    for (int e = threadIdx.x; e < kNT * cols; e += kNThr) {
        const int t = e / cols, j = e - t * cols;
        dst[t * 33 + j] = t < rows ? to_f32(src[t * ld + j]) : 0.0f;
    }
}
// a k x n matrix (row-major) -> dst[i * 33 + j]
template <typename E> __device__ __forceinline__ void stage_mat(const E *src, int k, int n, float *dst)
{
    for (int e = threadIdx.x; e < k * n; e += kNThr) {
        const int i = e / n;
        dst[i * 33 + e - i * n] = to_f32(src[e]);
    }
}

struct NarrowIn {
    const void *Z;        // T x d
    const void *W;        // element (c, j) at W[c * sk + j * sj]
    int64_t sk, sj, T, d;
    int m, r, act, merge;
    const void *V;        // encode: We2 (m x r); decode: Wd1 (r x m)
    const void *X;        // encode: X (T x d, null: P only); decode: B (T x r)
    void *out;            // encode: B; decode: dB (T x r)
    float *P;             // encode: P (T x m) or null; decode: dQ (T x m)
    float *G;             // decode: phi(Q) (T x m)
};

struct NarrowInSmem {
    __align__(16) float zs[kNT][kNChunk + 4];
    float rows1[kNT * 33], rows2[kNT * 33], vs[kNW * 33];
};

// One tile. MP: m rounded up to 4, 8, 16 or 32; lane j + MP * s of a warp takes column j of tokens s, s + 32 / MP, ...
template <typename E, int MP, bool DEC> __device__ __forceinline__ void narrow_in_tile(const NarrowIn &a, int64_t tile, NarrowInSmem &sh)
{
    auto &zs = sh.zs;
    float *rows1 = sh.rows1, *rows2 = sh.rows2, *vs = sh.vs;
    float *part = &zs[0][0];   // [warp][token][column], once the products have read zs
    static_assert(kNThr / 32 * kNT * MP <= kNT * (kNChunk + 4), "the warps' parts fit in the staged rows");
    constexpr int TPW = 32 / MP, NA = kNT / TPW > 0 ? kNT / TPW : 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j = lane % MP, ts = lane / MP;
    const int64_t t0 = tile * kNT;
    const int nt = a.T - t0 < kNT ? (int)(a.T - t0) : kNT;
    const E *Z = static_cast<const E *>(a.Z) + t0 * a.d, *W = static_cast<const E *>(a.W);
    stage_mat(static_cast<const E *>(a.V), DEC ? a.r : a.m, DEC ? a.m : a.r, vs);
    if (DEC) stage_rows(static_cast<const E *>(a.X) + t0 * a.r, a.r, nt, a.r, rows1);
    float acc[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) acc[i] = 0.0f;
    for (int64_t c0 = 0; c0 < a.d; c0 += kNChunk) {
        const int nc = a.d - c0 < kNChunk ? (int)(a.d - c0) : kNChunk;
        const int nc4 = (nc + 3) & ~3;
        if (c0) __syncthreads();
        for (int t = warp; t < kNT; t += kNThr / 32)
#pragma unroll 8
            for (int c = lane; c < nc4; c += 32) zs[t][c] = (t < nt && c < nc) ? to_f32(Z[t * a.d + c0 + c]) : 0.0f;
        __syncthreads();
        // this warp's share of the chunk's columns, a multiple of four
        const int per = (nc4 / 4 + kNThr / 32 - 1) / (kNThr / 32) * 4;
        const int b = warp * per, e = b + per < nc4 ? b + per : nc4;
        const E *w = W + c0 * a.sk + (j < a.m ? j : 0) * a.sj;
#pragma unroll 4
        for (int c = b; c < e; c += 4) {
            float wv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) wv[q] = (j < a.m && c + q < nc) ? to_f32(w[(c + q) * a.sk]) : 0.0f;
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const float4 z = *reinterpret_cast<const float4 *>(&zs[(ts + TPW * i) & (kNT - 1)][c]);
                acc[i] = fmaf(z.x, wv[0], acc[i]);
                acc[i] = fmaf(z.y, wv[1], acc[i]);
                acc[i] = fmaf(z.z, wv[2], acc[i]);
                acc[i] = fmaf(z.w, wv[3], acc[i]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NA; ++i) part[(warp * kNT + ts + TPW * i) * MP + j] = acc[i];
    __syncthreads();
    // the warps' parts in order; then the rest of the op on the tile's m- and r-wide rows
    for (int e = tid; e < kNT * a.m; e += kNThr) {
        const int t = e / a.m, k = e - t * a.m;
        float p = part[t * MP + k];
#pragma unroll
        for (int w = 1; w < kNThr / 32; ++w) p += part[(w * kNT + t) * MP + k];
        if (!DEC) {   // P = F . We1, phi(P)
            if (a.P && t < nt) a.P[(t0 + t) * a.m + k] = p;
            rows2[t * 33 + k] = act_f(a.act, p);
        } else {      // Q = B . Wd1; G = phi(Q); dQ = dG * phi'(Q)
            float q = 0.0f;
            for (int i = 0; i < a.r; ++i) q = fmaf(rows1[t * 33 + i], vs[i * 33 + k], q);
            float g, dg;
            act_and_dact(a.act, q, g, dg);
            rows2[t * 33 + k] = p * dg;
            if (t < nt) {
                a.G[(t0 + t) * a.m + k] = g;
                a.P[(t0 + t) * a.m + k] = p * dg;
            }
        }
    }
    if (!DEC && !a.X) return;   // P only
    __syncthreads();
    for (int e = tid; e < nt * a.r; e += kNThr) {
        const int t = e / a.r, n = e - t * a.r;
        float s = 0.0f;
        if (!DEC) {   // B = X[:, :r] + phi(P) . We2
            for (int k = 0; k < a.m; ++k) s = fmaf(rows2[t * 33 + k], vs[k * 33 + n], s);
            s += to_f32(static_cast<const E *>(a.X)[(t0 + t) * a.d + n]);
        } else {      // dB = [merge] dY[:, :r] + dQ . Wd1^T
            for (int k = 0; k < a.m; ++k) s = fmaf(rows2[t * 33 + k], vs[n * 33 + k], s);
            if (a.merge) s += to_f32(Z[t * a.d + n]);
        }
        static_cast<E *>(a.out)[(t0 + t) * a.r + n] = from_f32<E>(s);
    }
}

template <typename E, int MP, bool DEC> __global__ void __launch_bounds__(kNThr) k_narrow_in(const NarrowIn a)
{
    __shared__ NarrowInSmem sh;
    griddep_wait();
    griddep_launch_dependents();
    narrow_in_tile<E, MP, DEC>(a, blockIdx.x, sh);
}

struct NarrowOut {
    const void *In;       // T x r: B (decode forward) or dB (encode backward)
    const void *V;        // Wd1 (r x m) or We2 (m x r)
    const void *W;        // element (j, c) at W[j * sj + c * sc]
    int64_t sj, sc, T, d;
    int m, r, act, merge;
    const float *P;       // encode backward: P (T x m)
    void *out;            // T x d: Y or dF
    void *dX;             // encode backward: dX (T x d) or null
    float *dP, *A;        // encode backward: T x m each
};

template <bool ENC> struct NarrowOutSmem {
    __align__(16) float gs[kNW][kNT];                // the m-wide rows, [j][token]
    float in[kNT * 33], vs[kNW * 33];
    float ws[ENC ? kNThr * 33 : 1];                  // ENC: this block's columns of W
};

// One tile and block of 256 columns, a thread per column. DC: 256, or 64 where d is no larger: the tile's tokens then
// go round the block's four groups of threads (the same sums).
template <typename E, bool ENC, int DC>
__device__ __forceinline__ void narrow_out_tile(const NarrowOut &a, int64_t tile, int64_t cblk, NarrowOutSmem<ENC> &sh)
{
    float *ws = sh.ws, *in = sh.in, *vs = sh.vs;
    auto &gs = sh.gs;
    const int tid = threadIdx.x;
    const int64_t t0 = tile * kNT, c0 = cblk * kNThr;
    const int nt = a.T - t0 < kNT ? (int)(a.T - t0) : kNT;
    const int nc = a.d - c0 < kNThr ? (int)(a.d - c0) : kNThr;
    const E *W = static_cast<const E *>(a.W);
    stage_mat(static_cast<const E *>(a.V), ENC ? a.m : a.r, ENC ? a.r : a.m, vs);
    stage_rows(static_cast<const E *>(a.In) + t0 * a.r, a.r, nt, a.r, in);
    if (ENC)   // We1 (d x m): contiguous rows of m
        for (int e = tid; e < nc * a.m; e += kNThr) {
            const int c = e / a.m;
            ws[c * 33 + e - c * a.m] = to_f32(W[c0 * a.sc + e]);
        }
    __syncthreads();
    for (int e = tid; e < kNT * a.m; e += kNThr) {
        const int t = e / a.m, k = e - t * a.m;
        float s = 0.0f;
        if (!ENC) {   // G = phi(B . Wd1)
            for (int i = 0; i < a.r; ++i) s = fmaf(in[t * 33 + i], vs[i * 33 + k], s);
            s = act_f(a.act, s);
        } else {      // dP = (dB . We2^T) * phi'(P), A = phi(P)
            for (int i = 0; i < a.r; ++i) s = fmaf(in[t * 33 + i], vs[k * 33 + i], s);
            float f = 0.0f, df = 0.0f;
            if (t < nt) act_and_dact(a.act, a.P[(t0 + t) * a.m + k], f, df);
            s *= df;
            if (cblk == 0 && t < nt) {
                a.dP[(t0 + t) * a.m + k] = s;
                a.A[(t0 + t) * a.m + k] = f;
            }
        }
        gs[k][t] = s;
    }
    if (ENC && a.dX && cblk == 0)   // dX[:, :r] += dB
        for (int e = tid; e < nt * a.r; e += kNThr) {
            const int t = e / a.r, n = e - t * a.r;
            E *x = static_cast<E *>(a.dX) + (t0 + t) * a.d + n;
            *x = from_f32<E>(to_f32(*x) + in[t * 33 + n]);
        }
    __syncthreads();
    constexpr int NTG = kNT / (kNThr / DC);   // this thread's tokens, from tb on
    const int cl = DC == kNThr ? tid : tid % DC, tb = DC == kNThr ? 0 : tid / DC * NTG;
    const int64_t c = c0 + cl;
    if (cl >= nc) return;
    float acc[NTG];
#pragma unroll
    for (int t = 0; t < NTG; ++t) acc[t] = 0.0f;
#pragma unroll 4
    for (int k = 0; k < a.m; ++k) {
        const float w = ENC ? ws[cl * 33 + k] : to_f32(W[k * a.sj + c]);
#pragma unroll
        for (int q = 0; q < NTG / 4; ++q) {
            const float4 g = *reinterpret_cast<const float4 *>(&gs[k][tb + 4 * q]);
            acc[4 * q] = fmaf(g.x, w, acc[4 * q]);
            acc[4 * q + 1] = fmaf(g.y, w, acc[4 * q + 1]);
            acc[4 * q + 2] = fmaf(g.z, w, acc[4 * q + 2]);
            acc[4 * q + 3] = fmaf(g.w, w, acc[4 * q + 3]);
        }
    }
    E *o = static_cast<E *>(a.out) + (t0 + tb) * a.d + c;
#pragma unroll
    for (int t = 0; t < NTG; ++t)
        if (tb + t < nt) {
            const float skip = (!ENC && a.merge && c < a.r) ? in[(tb + t) * 33 + c] : 0.0f;
            o[t * a.d] = from_f32<E>(skip + acc[t]);
        }
}

template <typename E, bool ENC, int DC> __global__ void __launch_bounds__(kNThr) k_narrow_out(const NarrowOut a)
{
    __shared__ NarrowOutSmem<ENC> sh;
    griddep_wait();
    griddep_launch_dependents();
    narrow_out_tile<E, ENC, DC>(a, blockIdx.x, blockIdx.y, sh);
}

// The step's two decoder ops in one launch (both read B only): blocks [0, tiles) run the backward's tiles, the
// rest the forward's
template <typename E, int MP> __global__ void __launch_bounds__(kNThr) k_narrow_dec(const NarrowOut o, const NarrowIn i, int tiles)
{
    __shared__ union {
        NarrowInSmem in;
        NarrowOutSmem<false> out;
    } sh;
    griddep_wait();
    griddep_launch_dependents();
    if ((int)blockIdx.x < tiles) {
        narrow_in_tile<E, MP, true>(i, blockIdx.x, sh.in);
    } else {
        const int64_t k = (int64_t)blockIdx.x - tiles;
        narrow_out_tile<E, false, kNThr>(o, k % tiles, k / tiles, sh.out);
    }
}

struct NarrowWgrad {
    const void *Z;        // T x d: dY or F
    const float *V;       // T x m: phi(Q) or dP
    float *out;           // the d x m gradient: element (c, j) at out[c * sc + j * sj]
    int64_t sc, sj, T, d;
    int m, r;
    const void *io;       // T x r (B or dB)
    const float *U;       // T x m (dQ or phi(P))
    float *small;         // decode: r x m = io^T . U; encode: m x r = U^T . io
    int small_mr;         // 1: m x r
};

// One backward op's two gradients, or (jobs == 2: the step) both ops', the clusters' first half the first op's.
// Within a job, blockIdx.x / 8: the cluster's 64 columns of the d x m gradient, or (the last) the small one
struct NarrowWgrads {
    NarrowWgrad job[2];
    int jobs;
};
template <typename E, int MP>
__global__ void __launch_bounds__(kNThr) k_narrow_wgrad(const NarrowWgrads w)
{
    const int per_job = (int)gridDim.x / w.jobs;   // CTAs
    const bool second = (int)blockIdx.x >= per_job;
    const NarrowWgrad &a = w.job[second ? 1 : 0];
    const int cta = (int)blockIdx.x - (second ? per_job : 0);
    constexpr int TC = 64;                                   // tokens staged at a time
    __shared__ __align__(16) float buf[4 * 64 * (MP + 1) > TC * (MP + 33) ? 4 * 64 * (MP + 1) : TC * (MP + 33)];
    float(*vs)[MP] = reinterpret_cast<float(*)[MP]>(buf);
    float(*us)[33] = reinterpret_cast<float(*)[33]>(buf + TC * MP);
    float(*red)[64][MP + 1] = reinterpret_cast<float(*)[64][MP + 1]>(buf);   // after the products
    __shared__ float slots[kNCl][kNW * kNW / kNCl];          // the owned sums from every rank
    const int tid = threadIdx.x;
    const int rank = (int)cluster_rank();
    const int64_t chunk = cta / kNCl;
    const bool is_small = chunk == per_job / kNCl - 1;
    const int64_t tb = a.T * rank / kNCl, te = a.T * (rank + 1) / kNCl;   // this CTA's tokens
    griddep_wait();
    griddep_launch_dependents();
    cluster_sync();   // every CTA runs before anything is written into it
    if (is_small) {
        // up to 32 x 32 sums, four per thread; element e = i * m + j
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        const int n = a.r * a.m;
        for (int64_t t0 = tb; t0 < te; t0 += TC) {
            const int nt = te - t0 < TC ? (int)(te - t0) : TC;
            __syncthreads();
            for (int e = tid; e < nt * a.m; e += kNThr) vs[e / a.m][e % a.m] = a.U[t0 * a.m + e];
            for (int e = tid; e < nt * a.r; e += kNThr) us[e / a.r][e % a.r] = to_f32(static_cast<const E *>(a.io)[t0 * a.r + e]);
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = tid + kNThr * q;
                if (e < n) {
                    const int i = e / a.m, k = e - i * a.m;
                    float s = 0.0f;   // each block's sum by itself: one chain of a rank's T / 8 tokens rounds more
                    for (int t = 0; t < nt; ++t) s = fmaf(us[t][i], vs[t][k], s);   // (T = 65536: 4.9e-7 against 1.5e-7)
                    acc[q] += s;
                }
            }
        }
        const int own = (n + kNCl - 1) / kNCl;   // elements per owner, at most 128
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + kNThr * q;
            if (e < n) st_cluster_f32(map_shared(smem_addr(&slots[rank][e % own]), (uint32_t)(e / own)), acc[q]);
        }
        cluster_sync();
        for (int x = tid; x < own; x += kNThr) {
            const int e = rank * own + x;
            if (e >= n) break;
            float s = slots[0][x];
#pragma unroll
            for (int p = 1; p < kNCl; ++p) s += slots[p][x];
            const int i = e / a.m, k = e - i * a.m;
            a.small[a.small_mr ? k * a.r + i : e] = s;
        }
        return;
    }
    const int cl = tid & 63, sub = tid >> 6;
    const int64_t c = chunk * 64 + cl;
    const E *Z = static_cast<const E *>(a.Z) + (c < a.d ? c : a.d - 1);
    float acc[MP];
#pragma unroll
    for (int k = 0; k < MP; ++k) acc[k] = 0.0f;
    for (int64_t t0 = tb; t0 < te; t0 += TC) {
        const int nt = te - t0 < TC ? (int)(te - t0) : TC;
        float z[TC / 4];   // this thread's 16 tokens, all loads in flight
#pragma unroll
        for (int i = 0; i < TC / 4; ++i) z[i] = sub * (TC / 4) + i < nt ? to_f32(Z[(t0 + sub * (TC / 4) + i) * a.d]) : 0.0f;
        __syncthreads();
        for (int e = tid; e < TC * MP; e += kNThr) {
            const int t = e / MP, k = e % MP;
            vs[t][k] = (t < nt && k < a.m) ? a.V[(t0 + t) * a.m + k] : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TC / 4; ++i) {
#pragma unroll
            for (int q = 0; q < MP / 4; ++q) {
                const float4 v = *reinterpret_cast<const float4 *>(&vs[sub * (TC / 4) + i][4 * q]);
                acc[4 * q] = fmaf(z[i], v.x, acc[4 * q]);
                acc[4 * q + 1] = fmaf(z[i], v.y, acc[4 * q + 1]);
                acc[4 * q + 2] = fmaf(z[i], v.z, acc[4 * q + 2]);
                acc[4 * q + 3] = fmaf(z[i], v.w, acc[4 * q + 3]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < MP; ++k) red[sub][cl][k] = acc[k];
    __syncthreads();
    // the four token quarters in order, then to the owner: rank o owns columns [8 o, 8 o + 8) of the 64,
    // four of them per exchange (the slots hold 4 x 32 sums from each rank)
    for (int half = 0; half < 2; ++half) {
        if (half) cluster_sync();   // the first half's slots have been read
        for (int e = tid; e < 32 * MP; e += kNThr) {
            const int x = e / MP, k = e % MP;                 // x-th of the 32 columns of this half
            const int col = (x / 4) * 8 + half * 4 + (x % 4);
            const float s = ((red[0][col][k] + red[1][col][k]) + red[2][col][k]) + red[3][col][k];
            st_cluster_f32(map_shared(smem_addr(&slots[rank][(x % 4) * MP + k]), (uint32_t)(x / 4)), s);
        }
        cluster_sync();
        for (int e = tid; e < 4 * MP; e += kNThr) {
            float s = slots[0][e];
#pragma unroll
            for (int p = 1; p < kNCl; ++p) s += slots[p][e];
            const int k = e % MP;
            const int64_t col = chunk * 64 + rank * 8 + half * 4 + e / MP;
            if (k < a.m && col < a.d) a.out[col * a.sc + k * a.sj] = s;
        }
    }
}

// ---- launches (programmatic dependent launch: each kernel waits for its predecessor itself) ------
template <typename A>
cudaError_t launch_narrow(void (*kernel)(A), dim3 grid, int cluster, const A &a, const Ctx &c)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kNThr);
    cfg.stream = c.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    count_launches(1);
    return e;
}

template <typename E, bool DEC> cudaError_t narrow_in(const NarrowIn &a, const Ctx &c)
{
    const dim3 grid((unsigned)((a.T + kNT - 1) / kNT));
    return a.m <= 4    ? launch_narrow(k_narrow_in<E, 4, DEC>, grid, 1, a, c)
           : a.m <= 8  ? launch_narrow(k_narrow_in<E, 8, DEC>, grid, 1, a, c)
           : a.m <= 16 ? launch_narrow(k_narrow_in<E, 16, DEC>, grid, 1, a, c)
                       : launch_narrow(k_narrow_in<E, 32, DEC>, grid, 1, a, c);
}
// (rows of up to 64: fp32 m = 32 decoder forward T = 16384, d = 64 18.1 us with 256 columns a block, 12.4 with 64;
// 33 columns 17.8 and 12.3; T = 100 3.8 and 3.2. Of 65 to 255 columns a block of 256 leaves fewer threads idle)
template <typename E, bool ENC> cudaError_t narrow_out(const NarrowOut &a, const Ctx &c)
{
    const dim3 grid((unsigned)((a.T + kNT - 1) / kNT), (unsigned)((a.d + kNThr - 1) / kNThr));
    return a.d <= 64 ? launch_narrow(k_narrow_out<E, ENC, 64>, grid, 1, a, c)
                     : launch_narrow(k_narrow_out<E, ENC, kNThr>, grid, 1, a, c);
}
template <typename E> cudaError_t narrow_wgrad(const NarrowWgrads &w, const Ctx &c)
{
    const NarrowWgrad &a = w.job[0];
    const dim3 grid((unsigned)(w.jobs * kNCl * ((a.d + 63) / 64 + 1)));
    return a.m <= 4    ? launch_narrow(k_narrow_wgrad<E, 4>, grid, kNCl, w, c)
           : a.m <= 8  ? launch_narrow(k_narrow_wgrad<E, 8>, grid, kNCl, w, c)
           : a.m <= 16 ? launch_narrow(k_narrow_wgrad<E, 16>, grid, kNCl, w, c)
                       : launch_narrow(k_narrow_wgrad<E, 32>, grid, kNCl, w, c);
}

// ---- each op's arguments --------------------------------------------------------------------------
template <typename E>
NarrowIn narrow_enc_in(const resbm_desc &d, const E *X, const E *F, const E *We1, const E *We2, E *B, float *P)
{
    NarrowIn a{};
    a.Z = F; a.W = We1; a.sk = d.m; a.sj = 1; a.T = d.T; a.d = d.d;
    a.m = (int)d.m; a.r = (int)d.r; a.act = d.act;
    a.V = We2; a.X = X; a.out = B; a.P = P;
    return a;
}
template <typename E> NarrowOut narrow_dec_out(const resbm_desc &d, const E *B, const E *Wd1, const E *Wd2, E *Y)
{
    NarrowOut a{};
    a.In = B; a.V = Wd1; a.W = Wd2; a.sj = d.d; a.sc = 1; a.T = d.T; a.d = d.d;
    a.m = (int)d.m; a.r = (int)d.r; a.act = d.act; a.merge = d.merge_identity;
    a.out = Y;
    return a;
}
template <typename E>
NarrowIn narrow_dec_in(const resbm_desc &d, const E *dY, const E *B, const E *Wd1, const E *Wd2, E *dB, float *G, float *dQ)
{
    NarrowIn a{};
    a.Z = dY; a.W = Wd2; a.sk = 1; a.sj = d.d; a.T = d.T; a.d = d.d;
    a.m = (int)d.m; a.r = (int)d.r; a.act = d.act; a.merge = d.merge_identity;
    a.V = Wd1; a.X = B; a.out = dB; a.P = dQ; a.G = G;
    return a;
}
template <typename E>
NarrowWgrad narrow_dec_wgrad(const resbm_desc &d, const E *dY, const E *B, const float *G, const float *dQ, float *dWd1, float *dWd2)
{
    NarrowWgrad w{};
    w.Z = dY; w.V = G; w.out = dWd2; w.sc = 1; w.sj = d.d; w.T = d.T; w.d = d.d; w.m = (int)d.m; w.r = (int)d.r;
    w.io = B; w.U = dQ; w.small = dWd1; w.small_mr = 0;
    return w;
}
template <typename E>
NarrowOut narrow_enc_out(const resbm_desc &d, const E *dB, const float *P, const E *We1, const E *We2, E *dF, E *dX, float *dP,
                         float *A)
{
    NarrowOut a{};
    a.In = dB; a.V = We2; a.W = We1; a.sj = 1; a.sc = d.m; a.T = d.T; a.d = d.d;
    a.m = (int)d.m; a.r = (int)d.r; a.act = d.act;
    a.P = P; a.out = dF; a.dX = dX; a.dP = dP; a.A = A;
    return a;
}
template <typename E>
NarrowWgrad narrow_enc_wgrad(const resbm_desc &d, const E *F, const E *dB, const float *dP, const float *A, float *dWe1, float *dWe2)
{
    NarrowWgrad w{};
    w.Z = F; w.V = dP; w.out = dWe1; w.sc = d.m; w.sj = 1; w.T = d.T; w.d = d.d; w.m = (int)d.m; w.r = (int)d.r;
    w.io = dB; w.U = A; w.small = dWe2; w.small_mr = 1;
    return w;
}

// ---- the ops, and the step ---------------------------------------------------------------------------
template <typename E>
cudaError_t narrow_encode_fwd(const resbm_desc &d, const E *X, const E *F, const E *We1, const E *We2, E *B, float *P,
                              const Ctx &c)
{
    return narrow_in<E, false>(narrow_enc_in(d, X, F, We1, We2, B, P), c);
}
template <typename E>
cudaError_t narrow_decode_fwd(const resbm_desc &d, const E *B, const E *Wd1, const E *Wd2, E *Y, const Ctx &c)
{
    return narrow_out<E, false>(narrow_dec_out(d, B, Wd1, Wd2, Y), c);
}
// G, dQ: T x m fp32 scratch
template <typename E>
cudaError_t narrow_decode_bwd(const resbm_desc &d, const E *dY, const E *B, const E *Wd1, const E *Wd2, E *dB, float *dWd1,
                              float *dWd2, float *G, float *dQ, const Ctx &c)
{
    const cudaError_t e = narrow_in<E, true>(narrow_dec_in(d, dY, B, Wd1, Wd2, dB, G, dQ), c);
    if (e != cudaSuccess) return e;
    return narrow_wgrad<E>(NarrowWgrads{{narrow_dec_wgrad(d, dY, B, G, dQ, dWd1, dWd2), {}}, 1}, c);
}
// dP, A: T x m fp32 scratch
template <typename E>
cudaError_t narrow_encode_bwd(const resbm_desc &d, const E *dB, const E *F, const float *P, const E *We1, const E *We2,
                              E *dF, E *dX, float *dWe1, float *dWe2, float *dP, float *A, const Ctx &c)
{
    const cudaError_t e = narrow_out<E, true>(narrow_enc_out(d, dB, P, We1, We2, dF, dX, dP, A), c);
    if (e != cudaSuccess) return e;
    return narrow_wgrad<E>(NarrowWgrads{{narrow_enc_wgrad(d, F, dB, dP, A, dWe1, dWe2), {}}, 1}, c);
}
// The four ops in four launches instead of six (every output the same bits): the decoder's forward and
// backward together, and all four weight gradients. Small steps are launches and their latency: T = 512,
// d = 256, r = 2 fp32 20 us of GPU time and 11 us of enqueueing in six. scratch: four T x m fp32 matrices.
template <typename E>
cudaError_t narrow_step(const resbm_desc &d, const E *X, const E *F, const E *dY, const E *We1, const E *We2, const E *Wd1,
                        const E *Wd2, E *B, float *P, E *Y, E *dB, E *dF, E *dX, float *dWe1, float *dWe2, float *dWd1,
                        float *dWd2, float *const (&scratch)[4], const Ctx &c)
{
    float *G = scratch[0], *dQ = scratch[1], *dP = scratch[2], *A = scratch[3];
    cudaError_t e = narrow_encode_fwd<E>(d, X, F, We1, We2, B, P, c);
    if (e != cudaSuccess) return e;
    const NarrowOut o = narrow_dec_out(d, B, Wd1, Wd2, Y);
    const NarrowIn i = narrow_dec_in(d, dY, B, Wd1, Wd2, dB, G, dQ);
    const int tiles = (int)((d.T + kNT - 1) / kNT);
    const dim3 grid((unsigned)(tiles * (1 + (d.d + kNThr - 1) / kNThr)));
    auto kernel = d.m <= 4 ? k_narrow_dec<E, 4> : d.m <= 8 ? k_narrow_dec<E, 8> : d.m <= 16 ? k_narrow_dec<E, 16> : k_narrow_dec<E, 32>;
    e = launch_pdl(kernel, grid, dim3(kNThr), 0, c, o, i, tiles);
    count_launches(1);
    if (e == cudaSuccess) e = narrow_out<E, true>(narrow_enc_out(d, dB, P, We1, We2, dF, dX, dP, A), c);
    if (e != cudaSuccess) return e;
    return narrow_wgrad<E>(
        NarrowWgrads{{narrow_dec_wgrad(d, dY, B, G, dQ, dWd1, dWd2), narrow_enc_wgrad(d, F, dB, dP, A, dWe1, dWe2)}, 2}, c);
}

}  // namespace
}  // namespace resbm
