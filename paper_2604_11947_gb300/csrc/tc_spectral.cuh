// tc_spectral.cuh -- small kernels of the two matrix utilities around the bottleneck weights
// (Sec. 3.4.2 and the appendix's spectral analysis): the Frobenius normalisation that starts
// Muon's Newton-Schulz orthogonalisation, and the top eigenvalue of a Gram matrix W^T W by power
// iteration for the effective rank r_eff = sum sigma_i^2 / max sigma_i^2 = trace(W^T W) /
// lambda_max(W^T W). The products themselves run on the tensor-core GEMM (tc_gemm.cuh).
// Every sum here has a fixed order (per-block ranges, then the blocks in order): results are
// bitwise reproducible.
#pragma once

#include "common.cuh"
#include "tc_common.cuh"

namespace resbm {
namespace tc {

constexpr int kSqBlocks = 256;   // blocks of the sum-of-squares pass (fixed: a fixed summation order)

template <typename T> __device__ __forceinline__ float ld_f(const T *p, int64_t i) { return to_f32(p[i]); }

// part[b] = sum of x[i]^2 over block b's contiguous range (fp64), b < gridDim.x = kSqBlocks
template <typename T>
__global__ void __launch_bounds__(256) k_sumsq(const T *__restrict__ x, int64_t n, double *__restrict__ part)
{
    __shared__ double red[256];
    griddep_wait();
    griddep_launch_dependents();
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = blockIdx.x * per, b1 = b0 + per < n ? b0 + per : n;
    double s = 0.0;
    for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) {
        const double v = ld_f(x, i);
        s = fma(v, v, s);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// y = bf16(x / (||x||_F + eps)), ||x||_F^2 the sum of the kSqBlocks partials in a fixed order
template <typename T>
__global__ void __launch_bounds__(256) k_scale_bf16(const T *__restrict__ x, int64_t n, const double *__restrict__ part,
                                                    float eps, __nv_bfloat16 *__restrict__ y)
{
    __shared__ double red[kSqBlocks / 32];
    griddep_wait();
    griddep_launch_dependents();
    // one partial per thread, a fixed shuffle tree, then the warps in order (all partials in one chain
    // of dependent loads took 80 us of an 83 us launch at 4096 x 32)
    static_assert(kSqBlocks == 256, "one partial per thread");
    double s = part[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0.0;
#pragma unroll
    for (int w = 0; w < kSqBlocks / 32; ++w) s += red[w];
    const float inv = (float)(1.0 / (sqrt(s) + (double)eps));
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(ld_f(x, i) * inv);
}

// ---- Newton-Schulz in one launch for a small side of up to 64 -----------------------------------
// The whole iteration X <- a X + (b A + c A A) X, A = X X^T, on one cluster: CTA k keeps `lc` columns
// of the wide orientation of X (sd x ld, sd = min(rows, cols)) in shared memory as bf16 for all
// steps. Per step each CTA forms its partial Gram matrix (fp32), the cluster sums the partials in
// rank order (rank k owns 1 / cl of the elements, rounds its sums to bf16 and hands them to every
// CTA), and each CTA computes B = b A + c A A and its own columns of the next X. Every product has
// bf16 operands and fp32 accumulation and every iterate is rounded to bf16, as in the chain of
// GEMMs that takes the larger matrices.
// What bounds it: latency. A 4096 x 32 matrix is 256 KB and a step 8 MFLOP, nothing to the chip;
// the chain spent 17 launches on it, its Gram product one CTA walking all 4096 columns (19 us a
// step). Here a step costs two cluster exchanges and ~0.5 us of products. The products are
// m16n8k16 warp MMAs: tcgen05's 128-row tile would be three quarters padding and its results would
// have to come back from TMEM to registers at every step.
constexpr int kNsMaxSd = 64, kNsThreads = 256, kNsMaxCl = 8;
constexpr uint32_t kNsMaxSmem = 224 * 1024;

struct NsLayout {   // dynamic shared memory, byte offsets
    int cl, lc;     // CTAs, columns per CTA (a multiple of 64)
    uint32_t xs, as;   // row pitches of X and of A, B in bytes (16 bytes of padding: conflict-free ldmatrix)
    uint32_t x, a, b, red, slots, bytes;
};
__host__ __device__ inline NsLayout ns_layout(int sdp, int64_t ld)
{
    NsLayout l;
    l.cl = ld <= 64 ? 1 : ld <= 128 ? 2 : ld <= 256 ? 4 : 8;
    l.lc = (int)(((ld + l.cl - 1) / l.cl + 63) / 64 * 64);
    l.xs = (uint32_t)l.lc * 2 + 16;
    l.as = (uint32_t)sdp * 2 + 16;
    l.x = 0;
    l.a = l.x + (uint32_t)sdp * l.xs;
    l.b = l.a + (uint32_t)sdp * l.as;
    l.red = l.b + (uint32_t)sdp * l.as;                      // two partial Gram matrices
    l.slots = l.red + 2u * (uint32_t)(sdp * sdp) * 4;        // the owned elements from every rank
    l.bytes = l.slots + (uint32_t)(sdp * sdp) * 4;
    return l;
}
inline int ns_sdp(int64_t sd) { return (int)((sd + 15) / 16 * 16); }
inline bool ns_fused_ok(int64_t rows, int64_t cols)
{
    const int64_t sd = rows < cols ? rows : cols, ld = rows < cols ? cols : rows;
    return sd <= kNsMaxSd && ld <= (1 << 20) && ns_layout(ns_sdp(sd), ld).bytes <= kNsMaxSmem;
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

// SDP: sd rounded up to 16 (the padding rows and columns of X are zeros and stay zeros)
template <int SDP, typename TG>
__global__ void __launch_bounds__(kNsThreads, 1)
    k_newton_schulz(const TG *__restrict__ G, int sd, int64_t ld, int tall, int steps, float ca, float cb, float cc,
                    float eps, __nv_bfloat16 *__restrict__ out)
{
    extern __shared__ float4 ns_smem4[];
    uint8_t *sm = reinterpret_cast<uint8_t *>(ns_smem4);
    __shared__ double red[kNsThreads / 32], nslot[kNsMaxCl];
    const NsLayout L = ns_layout(SDP, ld);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = L.cl > 1 ? (int)cluster_rank() : 0;
    const int64_t l0 = (int64_t)rank * L.lc;
    const int nl = ld - l0 < 0 ? 0 : ld - l0 < L.lc ? (int)(ld - l0) : L.lc;   // this CTA's real columns
    griddep_wait();
    griddep_launch_dependents();
    auto sync_all = [&] {
        if (L.cl > 1) cluster_sync();
        else __syncthreads();
    };
    // element e of this CTA's part in memory order: (row i, column l) of the wide orientation
    const int ne = sd * nl;
    auto place = [&](int e, int &i, int &l) -> int64_t {
        if (tall) {
            l = e / sd;
            i = e - l * sd;
            return (l0 + l) * (int64_t)sd + i;
        }
        i = e / nl;
        l = e - i * nl;
        return (int64_t)i * ld + l0 + l;
    };
    // ||G||_F^2: squares in fp32 with their rounding errors carried along (two-term sums, ~2^-46
    // relative), or in fp64 where they leave fp32's range
    double s;
    {
        float hi = 0.0f, lo = 0.0f;
        for (int e = tid; e < ne; e += kNsThreads) {
            int i, l;
            const float v = to_f32(G[place(e, i, l)]);
            const float p = v * v, pe = fmaf(v, v, -p);
            const float t = hi + p, bb = t - hi;
            lo += (hi - (t - bb)) + (p - bb) + pe;
            hi = t;
        }
        s = (double)hi + (double)lo;
        if (!(hi < 1e37f)) {   // overflow (or NaN): again in fp64
            s = 0.0;
            for (int e = tid; e < ne; e += kNsThreads) {
                int i, l;
                const double v = to_f32(G[place(e, i, l)]);
                s = fma(v, v, s);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    // zero X's padding meanwhile (rows >= sd, columns >= nl)
    for (int e = tid; e < SDP * L.lc / 2; e += kNsThreads) {
        const int i = e / (L.lc / 2), l = 2 * (e % (L.lc / 2));
        if (i >= sd || l + 2 > nl) *reinterpret_cast<uint32_t *>(sm + L.x + i * L.xs + 2 * l) = 0u;
    }
    sync_all();   // every CTA runs before anything is written into it; red is complete
    if (tid < L.cl) {
        double t = 0.0;
        for (int w = 0; w < kNsThreads / 32; ++w) t += red[w];
        if (L.cl > 1)
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(map_shared(smem_u32(&nslot[rank]), (uint32_t)tid)), "d"(t)
                         : "memory");
        else
            nslot[0] = t;
    }
    sync_all();
    s = 0.0;
    for (int p = 0; p < L.cl; ++p) s += nslot[p];
    const float inv = (float)(1.0 / (sqrt(s) + (double)eps));
    for (int e = tid; e < ne; e += kNsThreads) {
        int i, l;
        const float v = to_f32(G[place(e, i, l)]);
        *reinterpret_cast<__nv_bfloat16 *>(sm + L.x + i * L.xs + 2 * l) = __float2bfloat16_rn(v * inv);
    }
    __syncthreads();

    const uint32_t xb = smem_u32(sm + L.x), ab = smem_u32(sm + L.a), bb = smem_u32(sm + L.b);
    float *gred = reinterpret_cast<float *>(sm + L.red);
    const float *slots = reinterpret_cast<const float *>(sm + L.slots);
    const int chunk = SDP * SDP / L.cl;
    const int kg = warp >> 1, nh = warp & 1;   // Gram: a quarter of the columns, half of the output columns
    constexpr int MT = SDP / 16, NTH = SDP / 16, NT8 = SDP / 8;
    for (int step = 0; step < steps; ++step) {
        // ---- this CTA's partial A = X X^T ----
        float acc[MT][NTH][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NTH; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.0f;
        for (int k0 = kg * (L.lc / 4); k0 < (kg + 1) * (L.lc / 4); k0 += 16) {
            uint32_t bf[NTH][2];
#pragma unroll
            for (int n = 0; n < NTH; ++n)
                ldsm2(bf[n], xb + (nh * (SDP / 2) + 8 * n + (lane & 7)) * L.xs + 2 * (k0 + 8 * ((lane >> 3) & 1)));
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                uint32_t af[4];
                ldsm4(af, xb + (16 * m + (lane & 15)) * L.xs + 2 * (k0 + 8 * (lane >> 4)));
#pragma unroll
                for (int n = 0; n < NTH; ++n) mma16816(acc[m][n], af, bf[n][0], bf[n][1]);
            }
        }
        auto each = [&](auto &&f) {   // f(element offset of a column pair, first value, second value)
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < NTH; ++n)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        f((16 * m + 8 * h + (lane >> 2)) * SDP + nh * (SDP / 2) + 8 * n + 2 * (lane & 3),
                          acc[m][n][2 * h], acc[m][n][2 * h + 1]);
        };
        // the four column quarters, pairwise: (0 + 2) + (1 + 3)
        if (kg >= 2) each([&](int o, float &a, float &b) { *reinterpret_cast<float2 *>(gred + (kg - 2) * SDP * SDP + o) = make_float2(a, b); });
        __syncthreads();
        if (kg < 2)
            each([&](int o, float &a, float &b) {
                const float2 t = *reinterpret_cast<const float2 *>(gred + kg * SDP * SDP + o);
                a += t.x;
                b += t.y;
            });
        if (kg == 1) each([&](int o, float &a, float &b) { *reinterpret_cast<float2 *>(gred + SDP * SDP + o) = make_float2(a, b); });
        __syncthreads();
        // to the owners of the elements
        if (kg == 0)
            each([&](int o, float &a, float &b) {
                const float2 t = *reinterpret_cast<const float2 *>(gred + SDP * SDP + o);
                const int owner = o / chunk;
                const uint32_t dst = smem_u32(sm + L.slots) + 4u * (uint32_t)(rank * chunk + o - owner * chunk);
                asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(map_shared(dst, (uint32_t)owner)),
                             "f"(a + t.x), "f"(b + t.y)
                             : "memory");
            });
        sync_all();
        // the owned sums, in rank order, rounded to bf16, to every CTA
        for (int e = tid; e < chunk / 2; e += kNsThreads) {
            float2 t = *reinterpret_cast<const float2 *>(slots + 2 * e);
            for (int p = 1; p < L.cl; ++p) {
                const float2 u = *reinterpret_cast<const float2 *>(slots + p * chunk + 2 * e);
                t.x += u.x;
                t.y += u.y;
            }
            const uint32_t v = pack_bf16(t.x, t.y);
            const int o = rank * chunk + 2 * e;
            const uint32_t dst = ab + (uint32_t)(o / SDP) * L.as + 2u * (uint32_t)(o % SDP);
            for (int p = 0; p < L.cl; ++p)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_shared(dst, (uint32_t)p)), "r"(v) : "memory");
        }
        sync_all();
        // ---- B = b A + c A A ----
        for (int t = warp; t < MT * NTH; t += kNsThreads / 32) {   // a 16 x 16 tile per warp
            const int m = t / NTH, n = t % NTH;
            float c0[4] = {0, 0, 0, 0}, c1[4] = {0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < MT; ++k) {
                uint32_t af[4], bf[4];
                ldsm4(af, ab + (16 * m + (lane & 15)) * L.as + 2 * (16 * k + 8 * (lane >> 4)));
                ldsm4t(bf, ab + (16 * k + (lane & 15)) * L.as + 2 * (16 * n + 8 * (lane >> 4)));
                mma16816(c0, af, bf[0], bf[1]);
                mma16816(c1, af, bf[2], bf[3]);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float *c = q ? c1 : c0;
                    const uint32_t o = (uint32_t)(16 * m + 8 * h + (lane >> 2)) * L.as + 2u * (uint32_t)(16 * n + 8 * q + 2 * (lane & 3));
                    const uint32_t a2 = *reinterpret_cast<const uint32_t *>(sm + L.a + o);
                    *reinterpret_cast<uint32_t *>(sm + L.b + o) =
                        pack_bf16(fmaf(cc, c[2 * h], cb * __uint_as_float(a2 << 16)),
                                  fmaf(cc, c[2 * h + 1], cb * __uint_as_float(a2 & 0xFFFF0000u)));
                }
        }
        __syncthreads();
        // ---- X <- a X + B X, 16 columns per warp at a time, in place ----
        for (int c0 = 16 * warp; c0 < L.lc; c0 += 16 * (kNsThreads / 32)) {
            uint32_t bf[MT][4];
#pragma unroll
            for (int k = 0; k < MT; ++k) ldsm4t(bf[k], xb + (16 * k + (lane & 15)) * L.xs + 2 * (c0 + 8 * (lane >> 4)));
            __syncwarp();
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                float d0[4] = {0, 0, 0, 0}, d1[4] = {0, 0, 0, 0};
#pragma unroll
                for (int k = 0; k < MT; ++k) {
                    uint32_t af[4];
                    ldsm4(af, bb + (16 * m + (lane & 15)) * L.as + 2 * (16 * k + 8 * (lane >> 4)));
                    mma16816(d0, af, bf[k][0], bf[k][1]);
                    mma16816(d1, af, bf[k][2], bf[k][3]);
                }
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float *d = q ? d1 : d0;
                        uint32_t *x = reinterpret_cast<uint32_t *>(sm + L.x + (16 * m + 8 * h + (lane >> 2)) * L.xs + 2 * (c0 + 8 * q + 2 * (lane & 3)));
                        *x = pack_bf16(fmaf(ca, __uint_as_float(*x << 16), d[2 * h]),
                                       fmaf(ca, __uint_as_float(*x & 0xFFFF0000u), d[2 * h + 1]));
                    }
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < ne; e += kNsThreads) {
        int i, l;
        const int64_t at = place(e, i, l);
        out[at] = *reinterpret_cast<const __nv_bfloat16 *>(sm + L.x + i * L.xs + 2 * l);
    }
    sync_all();   // no CTA leaves while another may still write into it
}

// Power iteration on a symmetric positive semi-definite n x n fp32 matrix G (row-major) by one
// CTA: v <- G v / ||G v|| from a fixed start vector, until the residual ||G v - lambda v|| of the
// Rayleigh quotient lambda = v^T G v (||v|| = 1) is at most tol * lambda, or max_iter iterations.
// For a symmetric matrix some eigenvalue lies within the residual of lambda (Bauer-Fike), so the
// stop bounds the eigenvalue's relative error by tol even when the top eigenvalues are close
// (where the Rayleigh quotient itself creeps slowly). out[0] = lambda_max,
// out[1] = trace(G) (fp64 sum in index order), out[2] = trace / lambda_max (the effective rank
// when G = W^T W), out[3] = iterations taken. The vectors live in shared memory (n <= kPowMaxN).
constexpr int kPowMaxN = 4096;
__global__ void __launch_bounds__(1024) k_power_iter(const float *__restrict__ G, int n, int max_iter, float tol,
                                                     double *__restrict__ out)
{
    __shared__ float v[kPowMaxN], y[kPowMaxN];
    __shared__ double red[32];
    __shared__ double bc;
    griddep_wait();
    griddep_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    // a fixed start with no special direction: 1 + 0.5 sin(0.7 j)
    for (int j = tid; j < n; j += blockDim.x) v[j] = 1.0f + 0.5f * sinf(0.7f * (float)j);
    __syncthreads();
    // block-wide sum of per-thread doubles in a fixed order
    auto block_sum = [&](double t) -> double {
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) red[warp] = t;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) s += red[w];
            bc = s;
        }
        __syncthreads();
        const double r = bc;
        __syncthreads();
        return r;
    };
    double nv = 0.0;
    for (int j = tid; j < n; j += blockDim.x) nv += (double)v[j] * v[j];
    nv = block_sum(nv);
    const float s0 = (float)(1.0 / sqrt(nv));
    for (int j = tid; j < n; j += blockDim.x) v[j] *= s0;
    __syncthreads();
    double lam = 0.0;
    int it = 0;
    for (; it < max_iter; ++it) {
        // y = G v: one warp per row, lanes along the row, a fixed reduction tree
        for (int i = warp; i < n; i += nw) {
            float acc = 0.0f;
            for (int j = lane; j < n; j += 32) acc = fmaf(G[(int64_t)i * n + j], v[j], acc);
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) y[i] = acc;
        }
        __syncthreads();
        double rq = 0.0, ny = 0.0, vv = 0.0;
        for (int j = tid; j < n; j += blockDim.x) {
            rq += (double)v[j] * y[j];
            ny += (double)y[j] * y[j];
            vv += (double)v[j] * v[j];
        }
        rq = block_sum(rq);
        ny = block_sum(ny);
        vv = block_sum(vv);
        lam = rq / vv;   // the Rayleigh quotient of v (unit length up to fp32 rounding)
        if (ny <= 0.0) break;   // G v = 0: G is zero on the start vector's span
        // the residual ||G v - lam v|| / ||v||, summed element by element in fp64
        double r2 = 0.0;
        for (int j = tid; j < n; j += blockDim.x) {
            const double t = (double)y[j] - lam * (double)v[j];
            r2 += t * t;
        }
        const double res = sqrt(block_sum(r2) / vv);
        const float s = (float)(1.0 / sqrt(ny));
        for (int j = tid; j < n; j += blockDim.x) v[j] = y[j] * s;
        __syncthreads();
        if (res <= (double)tol * fabs(lam)) {
            ++it;
            break;
        }
    }
    if (tid == 0) {
        double tr = 0.0;
        for (int i = 0; i < n; ++i) tr += (double)G[(int64_t)i * n + i];
        out[0] = lam;
        out[1] = tr;
        out[2] = lam > 0.0 ? tr / lam : 0.0;
        out[3] = (double)it;
    }
}

}  // namespace tc
}  // namespace resbm
