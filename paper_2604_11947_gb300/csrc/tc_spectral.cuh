// tc_spectral.cuh -- small kernels of the two matrix utilities around the bottleneck weights
// (Sec. 3.4.2 and the appendix's spectral analysis): the Frobenius normalisation that starts
// Muon's Newton-Schulz orthogonalisation, and the top eigenvalue of a Gram matrix W^T W by
// restarted Lanczos for the effective rank r_eff = sum sigma_i^2 / max sigma_i^2 = trace(W^T W) /
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
    // (one thread's square root and division: fp64 units are few, 256 threads' took 10 us)
    __shared__ float inv_sh;
    if (threadIdx.x == 0) {
        s = 0.0;
        for (int w = 0; w < kSqBlocks / 32; ++w) s += red[w];
        inv_sh = (float)(1.0 / (sqrt(s) + (double)eps));
    }
    __syncthreads();
    const float inv = inv_sh;
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

// four consecutive elements as fp32
__device__ __forceinline__ float4 ns_load4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 ns_load4(const __nv_bfloat16 *p)
{
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xFFFF0000u));
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
    // four consecutive elements of this CTA's part in memory order (sd, ld and nl are multiples of 8):
    // tall, row i .. i + 3 of column l of the wide orientation; wide, row i, columns l .. l + 3
    const int nq = sd * nl / 4;
    auto place = [&](int e, int &i, int &l) -> int64_t {
        const int per = (tall ? sd : nl) / 4;
        const int a = e / per, b = 4 * (e - a * per);
        i = tall ? b : a;
        l = tall ? a : b;
        return tall ? (l0 + l) * (int64_t)sd + i : (int64_t)i * ld + l0 + l;
    };
    auto load4 = [&](int e, int &i, int &l) { return ns_load4(G + place(e, i, l)); };
    // ||G||_F^2: squares in fp32 with their rounding errors carried along (two-term sums, ~2^-46
    // relative), or in fp64 where they leave fp32's range
    double s;
    {
        float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
        for (int e = tid; e < nq; e += kNsThreads) {
            int i, l;
            const float4 v4 = load4(e, i, l);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float p = v[k] * v[k], pe = fmaf(v[k], v[k], -p);
                const float t = hi + p, bb = t - hi;
                lo += (hi - (t - bb)) + (p - bb) + pe;
                hi = t;
            }
        }
        s = (double)hi + (double)lo;
        if (!(hi < 1e37f)) {   // overflow (or NaN): again in fp64
            s = 0.0;
            for (int e = tid; e < nq; e += kNsThreads) {
                int i, l;
                const float4 v = load4(e, i, l);
                s = fma((double)v.x, (double)v.x, s);
                s = fma((double)v.y, (double)v.y, s);
                s = fma((double)v.z, (double)v.z, s);
                s = fma((double)v.w, (double)v.w, s);
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
            st_cluster_f64(map_shared(smem_u32(&nslot[rank]), (uint32_t)tid), t);
        else
            nslot[0] = t;
    }
    sync_all();
    s = 0.0;
    for (int p = 0; p < L.cl; ++p) s += nslot[p];
    const float inv = (float)(1.0 / (sqrt(s) + (double)eps));
#pragma unroll 4
    for (int e = tid; e < nq; e += kNsThreads) {
        int i, l;
        const float4 v = load4(e, i, l);
        uint8_t *x = sm + L.x + i * L.xs + 2 * l;
        const uint32_t p01 = pack_bf16(v.x * inv, v.y * inv), p23 = pack_bf16(v.z * inv, v.w * inv);
        if (tall) {
            *reinterpret_cast<uint16_t *>(x) = (uint16_t)p01;
            *reinterpret_cast<uint16_t *>(x + L.xs) = (uint16_t)(p01 >> 16);
            *reinterpret_cast<uint16_t *>(x + 2 * L.xs) = (uint16_t)p23;
            *reinterpret_cast<uint16_t *>(x + 3 * L.xs) = (uint16_t)(p23 >> 16);
        } else {
            *reinterpret_cast<uint2 *>(x) = make_uint2(p01, p23);
        }
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
    for (int e = tid; e < nq; e += kNsThreads) {
        int i, l;
        const int64_t at = place(e, i, l);
        const uint8_t *x = sm + L.x + i * L.xs + 2 * l;
        uint2 v;
        if (tall) {
            auto get = [&](int k) { return (uint32_t) * reinterpret_cast<const uint16_t *>(x + k * L.xs); };
            v = make_uint2(get(0) | get(1) << 16, get(2) | get(3) << 16);
        } else {
            v = *reinterpret_cast<const uint2 *>(x);
        }
        *reinterpret_cast<uint2 *>(out + at) = v;
    }
    sync_all();   // no CTA leaves while another may still write into it
}

// The largest eigenvalue of a symmetric positive semi-definite n x n fp32 matrix G (row-major) by
// restarted Lanczos on one cluster of kLzCl CTAs. A cycle builds up to kLzK orthonormal vectors
// q_0 .. q_{k-1} (every new vector orthogonalised twice against all earlier ones of the cycle) and
// the tridiagonal projection of G on them; the cycle's top Ritz vector starts the next. Each cycle
// begins with the check that ends the iteration: with v the start vector, lambda = v^T G v / v^T v
// and the residual ||G v - lambda v|| / ||v|| (sums in fp64) at most tol * lambda. For a symmetric
// matrix some eigenvalue then lies within the residual of lambda (Bauer-Fike), also when the top
// eigenvalues are close. out[0] = lambda_max, out[1] = trace(G) (fp64), out[2] = trace / lambda_max
// (the effective rank when G = W^T W), out[3] = products with G taken.
//
// What bounds it: latency. A step is one product with G (each CTA's rows, held in shared memory
// where they fit: n = 512 is 128 KB a CTA) and three exchanges over the cluster (twice the
// projections on the earlier vectors; the norm together with the new vector). Power iteration on one CTA
// (the Gram matrix read from L2 by one SM, ~9 us a product) needed thousands of products where the
// top eigenvalues are close, Lanczos ~100. Measured at n = 512 (W 8192 x 512, random): 25-40 ms by
// power iteration, 0.65-0.71 ms by this kernel, 0.37 ms by k_lanczos_small, which takes n <= 512.
// Every CTA takes each decision from the same sums, added in rank order: the cluster stays in
// step, and results are bitwise reproducible.
constexpr int kPowMaxN = 4096;
constexpr int kLzCl = 8, kLzThreads = 512, kLzK = 32;
constexpr uint32_t kLzMaxSmem = 216 * 1024;   // beside ~6 KB of static shared memory

struct LanczosLayout {   // dynamic shared memory, in floats; rows: G's rows per CTA
    int rows, v, y, q, g, floats;
    bool g_in_smem;
};
__host__ __device__ inline LanczosLayout lanczos_layout(int n)
{
    LanczosLayout l;
    l.rows = ((n + kLzCl - 1) / kLzCl + 3) / 4 * 4;
    l.v = 0;                         // two full vectors
    l.y = 2 * n;                     // this CTA's part of the current product
    l.q = l.y + l.rows;              // this CTA's part of the cycle's vectors
    l.g = l.q + kLzK * l.rows;
    l.g_in_smem = (int64_t)l.g + (int64_t)l.rows * n <= (int64_t)kLzMaxSmem / 4;
    l.floats = l.g_in_smem ? l.g + l.rows * n : l.g;
    return l;
}

// The top eigenvector s (unnormalised) of the k x k tridiagonal matrix (diagonal a, off-diagonals
// b[1 .. k-1]), one warp: the top eigenvalue by 33-section with Sturm counts (the pivots of
// T - x I, one positive pivot per eigenvalue above x), then one step of inverse iteration from
// the upper end of the last interval by the twisted factorisation (forward and backward pivots
// meeting where they nearly cancel).
__device__ __forceinline__ void tridiag_top(const float *a, const float *b, int k, float *d, float *u, float *s)
{
    const int lane = threadIdx.x & 31;
    float lo = a[0], hi = a[0];
    for (int i = 0; i < k; ++i) {
        lo = fmaxf(lo, a[i]);
        hi = fmaxf(hi, a[i] + (i > 0 ? fabsf(b[i]) : 0.0f) + (i + 1 < k ? fabsf(b[i + 1]) : 0.0f));
    }
    const float tiny = 1e-30f + 1e-14f * fabsf(hi);
    hi += 1e-6f * fabsf(hi) + tiny;
    for (int round = 0; round < 5; ++round) {
        const float x = lo + (hi - lo) * ((float)(lane + 1) / 33.0f);
        float p = a[0] - x;
        bool above = p > 0.0f;
        for (int i = 1; i < k; ++i) {
            if (fabsf(p) < tiny) p = -tiny;
            p = a[i] - x - __fdividef(b[i] * b[i], p);
            above = above || p > 0.0f;
        }
        const unsigned m = __ballot_sync(0xffffffffu, above);
        const int top = m ? 31 - __clz((int)m) : -1;   // the highest shift below the eigenvalue
        const float nlo = lo + (hi - lo) * ((float)(top + 1) / 33.0f);
        hi = lo + (hi - lo) * ((float)(top + 2) / 33.0f);
        lo = nlo;
    }
    if (lane < 2) {   // lane 0: forward pivots d; lane 1: backward pivots u
        float p = 0.0f;
        for (int t = 0; t < k; ++t) {
            const int i = lane == 0 ? t : k - 1 - t;
            const float off = t == 0 ? 0.0f : lane == 0 ? b[i] : b[i + 1];
            p = a[i] - hi - (t == 0 ? 0.0f : off * off / p);
            if (fabsf(p) < tiny) p = -tiny;
            (lane == 0 ? d : u)[i] = p;
        }
    }
    __syncwarp();
    if (lane == 0) {
        int r = 0;
        float best = 3.4e38f;
        for (int i = 0; i < k; ++i) {
            const float g = fabsf(d[i] + u[i] - (a[i] - hi));
            if (g < best) { best = g; r = i; }
        }
        s[r] = 1.0f;
        for (int i = r; i > 0; --i) s[i - 1] = -b[i] / d[i - 1] * s[i];
        for (int i = r; i + 1 < k; ++i) s[i + 1] = -b[i + 1] / u[i + 1] * s[i];
    }
    __syncwarp();
}

// One warp: the cycle's top Ritz vector s after k vectors (tridiag_top), and in *stop whether its residual's estimate,
// the new direction's norm beta times its last component, is below half the stop.
__device__ __forceinline__ void ritz_converged(const float *a, const float *b, int k, float *d, float *u, float *s, float beta,
                                               float tol, float lam, int *stop)
{
    tridiag_top(a, b, k, d, u, s);
    if ((threadIdx.x & 31) == 0) {
        float s2 = 0.0f;
        for (int v = 0; v < k; ++v) s2 = fmaf(s[v], s[v], s2);
        *stop = beta * fabsf(s[k - 1]) <= 0.5f * tol * fabsf(lam) * sqrtf(s2);
    }
}

// The power of two that brings a Gram matrix's trace to about 1. Both kernels multiply their products with
// G by it: the sums of squares and the tridiagonal matrix, whose elements scale with sigma^4 where they are
// squared, then keep to fp32's range for every G that does itself (the effective rank does not depend on
// W's scale). Exact, and undone in fp64 in the results; 1 for a zero matrix, infinities and NaN.
__device__ __forceinline__ float gram_scale(double trace)
{
    if (!(trace > 0.0) || isinf(trace)) return 1.0f;
    const int e = ilogb(trace);
    return ldexpf(1.0f, e < -126 ? 126 : e > 126 ? -126 : -e);
}

// The form for n <= kLzSmallN: every CTA keeps the whole of the cycle's vectors and repeats their
// orthogonalisation, so that a step's only exchange is the product itself (each CTA's rows of G v into
// every CTA's copy). With the vectors spread over the cluster (k_lanczos_top) a step takes three
// exchanges with a remote store's round trip each: W 8192 x 512, 614 us a call against 370 us.
// A cycle also ends early when the residual estimate |beta s_k| of its top Ritz pair, taken after 8 and
// 16 vectors, is below half the stop.
constexpr int kLzSmallN = 512;
struct LanczosSmall {   // dynamic shared memory, in floats
    int rows, y, g, floats;
};
__host__ __device__ inline LanczosSmall lanczos_small(int n)
{
    LanczosSmall l;
    l.rows = ((n + kLzCl - 1) / kLzCl + 3) / 4 * 4;
    l.y = kLzK * n;          // after the cycle's vectors: the products, two buffers
    l.g = l.y + 2 * n;       // this CTA's rows of G
    l.floats = l.g + l.rows * n;
    return l;
}

__global__ void __launch_bounds__(kLzThreads, 1) k_lanczos_small(const float *__restrict__ G, int n, int max_iter, float tol,
                                                                 double *__restrict__ out)
{
    extern __shared__ float4 lz_smem4[];
    float *sm = reinterpret_cast<float *>(lz_smem4);
    constexpr int NW = kLzThreads / 32;
    __shared__ double red[3][NW];
    __shared__ float fred[NW], hs[kLzK], al[kLzK], be[kLzK + 1], sv[kLzK], pd[kLzK], pu[kLzK];
    __shared__ int stop_early;
    const LanczosSmall L = lanczos_small(n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster_rank(), row0 = rank * L.rows;
    const int nr = n - row0 < 0 ? 0 : n - row0 < L.rows ? n - row0 : L.rows;
    float *Q = sm;
    const float *Gr = sm + L.g;
    griddep_wait();
    griddep_launch_dependents();
    {
        const float4 *src = reinterpret_cast<const float4 *>(G + (int64_t)row0 * n);
        float4 *dst = reinterpret_cast<float4 *>(sm + L.g);
        for (int e = tid; e < nr * n / 4; e += kLzThreads) dst[e] = src[e];
    }
    // block-wide sums in a fixed order (a warp's tree, then the warps in order), on every thread
    auto sums = [&](auto &t) {
        constexpr int NV = sizeof(t) / sizeof(double);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            for (int o = 16; o > 0; o >>= 1) t[v] += __shfl_xor_sync(0xffffffffu, t[v], o);
            if (lane == 0) red[v][warp] = t[v];
        }
        __syncthreads();
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            t[v] = 0.0;
            for (int w = 0; w < NW; ++w) t[v] += red[v][w];
        }
        __syncthreads();
    };
    // (n <= kLzThreads: one element per thread)
    const bool on = tid < n;
    // a fixed start with no special direction: 1 + 0.5 sin(0.7 j); the trace from G itself
    double t2[2];
    float q = on ? 1.0f + 0.5f * sinf(0.7f * (float)tid) : 0.0f;
    t2[0] = on ? (double)G[(int64_t)tid * n + tid] : 0.0;
    t2[1] = (double)q * q;
    sums(t2);
    const double trace = t2[0];
    const float gs = gram_scale(trace);
    if (on) Q[tid] = q * (float)(1.0 / sqrt(t2[1]));
    cluster_sync();   // every CTA runs before anything is written into it (and Q, G are complete)

    const int kmax = n < kLzK ? n : kLzK;
    int j = 0, it = 0;
    uint32_t buf = 0;
    double lam = 0.0;
    for (;;) {
        // y = gs G q_j, one warp per four rows, every row's sum into all CTAs' copies
        {
            const float4 *v4 = reinterpret_cast<const float4 *>(Q + j * n);
            const uint32_t ydst = smem_u32(sm + L.y + buf * n);
            for (int i0 = 4 * warp; i0 < nr; i0 += 4 * NW) {
                const float4 *g4 = reinterpret_cast<const float4 *>(Gr + i0 * n);
                float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                const int last = nr - i0 - 1;
                for (int c = lane; c < n / 4; c += 32) {
                    const float4 x = v4[c];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float4 g = g4[(r < last ? r : last) * (n / 4) + c];
                        acc[r] = fmaf(g.x, x.x, fmaf(g.y, x.y, fmaf(g.z, x.z, fmaf(g.w, x.w, acc[r]))));
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
                const int r = lane & 3;   // eight CTAs x four rows
                if (r <= last)
                    st_cluster_f32(map_shared(ydst + 4u * (uint32_t)(row0 + i0 + r), (uint32_t)(lane >> 2)),
                                   gs * (r == 0 ? acc[0] : r == 1 ? acc[1] : r == 2 ? acc[2] : acc[3]));
            }
        }
        cluster_sync();
        float *y = sm + L.y + buf * n;
        buf ^= 1;
        float w = on ? y[tid] : 0.0f;   // this thread's element of the new direction
        if (j == 0) {   // lambda and the residual of the cycle's start vector
            const double v = on ? (double)Q[tid] : 0.0;
            double t3[3] = {v * w, (double)w * w, v * v};
            sums(t3);
            lam = t3[0] / t3[2];
            if (t3[1] <= 0.0) break;   // G v = 0: G is zero on the start vector's span
            if (!isfinite(lam)) {      // G holds infinities or NaN: no iteration changes that
                it = max_iter;
                break;
            }
            if (it < max_iter) ++it;
            // ||y - lam v||^2 from the three fp64 sums (their rounding, ~1e-16 lam^2, is far below tol^2 lam^2)
            const double r2 = t3[1] - 2.0 * lam * t3[0] + lam * lam * t3[2];
            if (sqrt((r2 > 0.0 ? r2 : 0.0) / t3[2]) <= (double)tol * fabs(lam) || it >= max_iter) break;
            if (tid == 0) al[0] = (float)lam;
            if (on) w = fmaf(-(float)lam, Q[tid], w);
        } else {
            // the projections on the cycle's vectors removed, twice (see k_lanczos_top)
            ++it;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                if (pass) {
                    if (on) y[tid] = w;
                    __syncthreads();
                }
                for (int v = warp; v <= j; v += NW) {
                    float h = 0.0f;
                    for (int i = lane; i < n; i += 32) h = fmaf(Q[v * n + i], y[i], h);
                    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
                    if (lane == 0) hs[v] = h;
                }
                __syncthreads();
                if (tid == 0) al[j] = pass ? al[j] + hs[j] : hs[j];
                if (on) {
                    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
                    int v = 0;
                    for (; v + 4 <= j + 1; v += 4) {
                        s0 = fmaf(hs[v], Q[v * n + tid], s0);
                        s1 = fmaf(hs[v + 1], Q[(v + 1) * n + tid], s1);
                        s2 = fmaf(hs[v + 2], Q[(v + 2) * n + tid], s2);
                        s3 = fmaf(hs[v + 3], Q[(v + 3) * n + tid], s3);
                    }
                    for (; v <= j; ++v) s0 = fmaf(hs[v], Q[v * n + tid], s0);
                    w -= (s0 + s1) + (s2 + s3);
                }
            }
        }
        float b2 = w * w;
        for (int o = 16; o > 0; o >>= 1) b2 += __shfl_xor_sync(0xffffffffu, b2, o);
        if (lane == 0) fred[warp] = b2;
        __syncthreads();
        b2 = 0.0f;
#pragma unroll
        for (int x = 0; x < NW; ++x) b2 += fred[x];
        const float beta = sqrtf(b2);
        bool more = j + 1 < kmax && it < max_iter && beta > 1e-6f * fabsf((float)lam);
        bool have_s = false;
        if (more && (j + 1 == 8 || j + 1 == 16)) {
            if (warp == 0) ritz_converged(al, be, j + 1, pd, pu, sv, beta, tol, (float)lam, &stop_early);
            __syncthreads();
            if (stop_early) {
                more = false;
                have_s = true;
            }
        }
        if (more) {
            if (tid == 0) be[j + 1] = beta;
            ++j;
            if (on) Q[j * n + tid] = w * (1.0f / beta);
            __syncthreads();
            continue;
        }
        // the cycle's top Ritz vector starts the next cycle
        if (!have_s) {
            if (warp == 0) tridiag_top(al, be, j + 1, pd, pu, sv);
            __syncthreads();
        }
        float z = 0.0f;
        if (on)
            for (int v = 0; v <= j; ++v) z = fmaf(sv[v], Q[v * n + tid], z);
        double t1[1] = {(double)z * z};
        sums(t1);
        if (on) Q[tid] = z * (float)(1.0 / sqrt(t1[0]));
        j = 0;
        __syncthreads();
    }
    if (rank == 0 && tid == 0) {
        lam /= (double)gs;
        out[0] = lam;
        out[1] = trace;
        out[2] = lam > 0.0 ? trace / lam : 0.0;
        out[3] = (double)it;
    }
    cluster_sync();   // no CTA leaves while another may still write into it
}

__global__ void __launch_bounds__(kLzThreads, 1) k_lanczos_top(const float *__restrict__ G, int n, int max_iter, float tol,
                                                               double *__restrict__ out)
{
    extern __shared__ float4 lz_smem4[];
    float *sm = reinterpret_cast<float *>(lz_smem4);
    __shared__ double slots[2][3][kLzCl];      // exchanged partial sums: [buffer][value][rank]
    __shared__ float hslots[2][kLzK][kLzCl];   // the same for the projections
    __shared__ double red[3][kLzThreads / 32];
    __shared__ float hs[kLzK], al[kLzK], be[kLzK + 1], sv[kLzK], pd[kLzK], pu[kLzK];
    __shared__ int stop_early;
    const LanczosLayout L = lanczos_layout(n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = kLzThreads / 32;
    const int rank = (int)cluster_rank();
    const int row0 = rank * L.rows;
    const int nr = n - row0 < 0 ? 0 : n - row0 < L.rows ? n - row0 : L.rows;
    float *y = sm + L.y, *Q = sm + L.q;
    griddep_wait();
    griddep_launch_dependents();

    const float *Gr = G + (int64_t)row0 * n;
    if (L.g_in_smem) {
        const float4 *src = reinterpret_cast<const float4 *>(Gr);
        float4 *dst = reinterpret_cast<float4 *>(sm + L.g);
        for (int e = tid; e < nr * n / 4; e += kLzThreads) dst[e] = src[e];
        Gr = sm + L.g;
    }
    // a fixed start with no special direction: 1 + 0.5 sin(0.7 j)
    for (int j = tid; j < n; j += kLzThreads) sm[j] = 1.0f + 0.5f * sinf(0.7f * (float)j);

    // sums of NV doubles over the block (warp tree, then the warps in order); valid in lane v < NV of warp 0
    auto block_sums = [&](auto &t) {
        constexpr int NV = sizeof(t) / sizeof(double);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            for (int o = 16; o > 0; o >>= 1) t[v] += __shfl_xor_sync(0xffffffffu, t[v], o);
            if (lane == 0) red[v][warp] = t[v];
        }
        __syncthreads();
        double r = 0.0;
        if (tid < NV)
            for (int w = 0; w < NW; ++w) r += red[tid][w];
        return r;
    };
    uint32_t buf = 0;   // exchange buffer of the next exchange
    auto send = [&](int v, double x, int to) {
        st_cluster_f64(map_shared(smem_u32(&slots[buf][v][rank]), (uint32_t)to), x);
    };
    auto total = [&](uint32_t b, int v) {
        double s = 0.0;
#pragma unroll
        for (int p = 0; p < kLzCl; ++p) s += slots[b][v][p];
        return s;
    };

    // the trace and the start vector's norm (this CTA's rows; exchanged over the cluster)
    __syncthreads();
    double t2[2] = {0.0, 0.0};
    for (int i = tid; i < nr; i += kLzThreads) {
        t2[0] += (double)Gr[(int64_t)i * n + row0 + i];
        t2[1] += (double)sm[row0 + i] * sm[row0 + i];
    }
    double bs = block_sums(t2);
    cluster_sync();   // every CTA runs before anything is written into it
    if (tid < 2)
        for (int p = 0; p < kLzCl; ++p) send(tid, bs, p);
    cluster_sync();
    const double trace = total(buf, 0);
    const float gs = gram_scale(trace);
    float scale = (float)(1.0 / sqrt(total(buf, 1)));   // 1 / ||v||: v is kept unnormalised
    buf ^= 1;
    for (int i = tid; i < nr; i += kLzThreads) Q[i] = sm[row0 + i] * scale;

    const int kmax = n < kLzK ? n : kLzK;
    int cur = 0, j = 0, it = 0;
    double lam = 0.0;
    for (;;) {
        __syncthreads();   // y of the previous step has been read
        // y = scale * gs G v, one warp per four rows
        {
            const float4 *v4 = reinterpret_cast<const float4 *>(sm + cur * n);
            for (int i0 = 4 * warp; i0 < nr; i0 += 4 * NW) {
                const float4 *g4 = reinterpret_cast<const float4 *>(Gr + (int64_t)i0 * n);
                float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                const int last = nr - i0 - 1;
                for (int c = lane; c < n / 4; c += 32) {
                    const float4 x = v4[c];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float4 g = g4[(int64_t)(r < last ? r : last) * (n / 4) + c];
                        acc[r] = fmaf(g.x, x.x, fmaf(g.y, x.y, fmaf(g.z, x.z, fmaf(g.w, x.w, acc[r]))));
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
                if (lane < 4 && lane <= last)
                    y[i0 + lane] = scale * (gs * (lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3]));
            }
        }
        __syncthreads();
        if (j == 0) {   // lambda and the residual of the cycle's start vector
            double t3[3] = {0.0, 0.0, 0.0};
            for (int i = tid; i < nr; i += kLzThreads) {
                const double v = Q[i], w = y[i];
                t3[0] = fma(v, w, t3[0]);
                t3[1] = fma(w, w, t3[1]);
                t3[2] = fma(v, v, t3[2]);
            }
            bs = block_sums(t3);
            if (tid < 3)
                for (int p = 0; p < kLzCl; ++p) send(tid, bs, p);
            cluster_sync();
            const double vy = total(buf, 0), yy = total(buf, 1), vv = total(buf, 2);
            buf ^= 1;
            lam = vy / vv;
            if (yy <= 0.0) break;   // G v = 0: G is zero on the start vector's span
            if (!isfinite(lam)) {   // G holds infinities or NaN: no iteration changes that
                it = max_iter;
                break;
            }
            if (it < max_iter) ++it;
            // ||y - lam v||^2 from the three fp64 sums (their rounding, ~1e-16 lam^2, is far below tol^2 lam^2)
            const double r2 = yy - 2.0 * lam * vy + lam * lam * vv;
            if (sqrt((r2 > 0.0 ? r2 : 0.0) / vv) <= (double)tol * fabs(lam) || it >= max_iter) break;
            if (tid == 0) al[0] = (float)lam;
            for (int i = tid; i < nr; i += kLzThreads) y[i] = fmaf(-(float)lam, Q[i], y[i]);
        } else {
            // the projections on the cycle's vectors removed (one warp per vector), twice: the vectors
            // are orthogonal to E ~ eps, one pass leaves E G q behind, which the division by the new
            // direction's norm (a tenth of ||G q|| for a flat spectrum) would let grow tenfold a step
            ++it;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                for (int v = warp; v <= j; v += NW) {
                    float h = 0.0f;
                    for (int i = lane; i < nr; i += 32) h = fmaf(Q[v * L.rows + i], y[i], h);
                    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
                    if (lane < kLzCl)
                        st_cluster_f32(map_shared(smem_u32(&hslots[pass][v][rank]), (uint32_t)lane), h);
                }
                cluster_sync();
                if (tid <= j) {
                    float h = 0.0f;
#pragma unroll
                    for (int p = 0; p < kLzCl; ++p) h += hslots[pass][tid][p];
                    hs[tid] = h;
                }
                __syncthreads();
                if (tid == 0) al[j] = pass ? al[j] + hs[j] : hs[j];
                // eight threads per row (n = 512: one row each), every eighth vector a thread
                for (int i = tid >> 3; i < L.rows; i += kLzThreads / 8) {
                    float w = 0.0f;
                    for (int v = tid & 7; v <= j; v += 8) w = fmaf(hs[v], Q[v * L.rows + i], w);
                    w += __shfl_xor_sync(0xffffffffu, w, 1);
                    w += __shfl_xor_sync(0xffffffffu, w, 2);
                    w += __shfl_xor_sync(0xffffffffu, w, 4);
                    if ((tid & 7) == 0 && i < nr) y[i] -= w;
                }
                __syncthreads();
            }
        }
        __syncthreads();
        // the new direction's norm, and the direction itself into every CTA's other vector
        double t1[1] = {0.0};
        for (int i = tid; i < nr; i += kLzThreads) t1[0] = fma((double)y[i], (double)y[i], t1[0]);
        bs = block_sums(t1);
        if (tid == 0)
            for (int p = 0; p < kLzCl; ++p) send(0, bs, p);
        const uint32_t vdst = smem_u32(sm + (cur ^ 1) * n + row0);
        for (int e = tid; e < nr * kLzCl; e += kLzThreads)
            st_cluster_f32(map_shared(vdst + 4u * (uint32_t)(e / kLzCl), (uint32_t)(e % kLzCl)), y[e / kLzCl]);
        cluster_sync();
        const float beta = (float)sqrt(total(buf, 0));
        buf ^= 1;
        bool more = j + 1 < kmax && it < max_iter && beta > 1e-6f * fabsf((float)lam), have_s = false;
        // an early end of the cycle as in k_lanczos_small, from 2 vectors on (a product costs more here): one
        // dominant singular value needs three (2048 x 520, all but rank one: 358 us by whole cycles)
        if (more && (j + 1 == 2 || j + 1 == 4 || j + 1 == 16)) {
            if (warp == 0) ritz_converged(al, be, j + 1, pd, pu, sv, beta, tol, (float)lam, &stop_early);
            __syncthreads();
            have_s = stop_early != 0;
            more = !have_s;
        }
        if (more) {
            if (tid == 0) be[j + 1] = beta;
            scale = 1.0f / beta;
            cur ^= 1;
            ++j;
            for (int i = tid; i < nr; i += kLzThreads) Q[j * L.rows + i] = y[i] * scale;
            continue;   // (Q and be are read after later barriers)
        }
        // the cycle's top Ritz vector starts the next cycle
        if (!have_s && warp == 0) tridiag_top(al, be, j + 1, pd, pu, sv);
        __syncthreads();
        t1[0] = 0.0;
        for (int i = tid; i < nr; i += kLzThreads) {
            float w = 0.0f;
            for (int v = 0; v <= j; ++v) w = fmaf(sv[v], Q[v * L.rows + i], w);
            y[i] = w;
            t1[0] = fma((double)w, (double)w, t1[0]);
        }
        bs = block_sums(t1);
        if (tid == 0)
            for (int p = 0; p < kLzCl; ++p) send(0, bs, p);
        for (int e = tid; e < nr * kLzCl; e += kLzThreads)
            st_cluster_f32(map_shared(vdst + 4u * (uint32_t)(e / kLzCl), (uint32_t)(e % kLzCl)), y[e / kLzCl]);
        cluster_sync();
        scale = (float)(1.0 / sqrt(total(buf, 0)));
        buf ^= 1;
        cur ^= 1;
        j = 0;
        for (int i = tid; i < nr; i += kLzThreads) Q[i] = y[i] * scale;
    }
    if (rank == 0 && tid == 0) {
        lam /= (double)gs;
        out[0] = lam;
        out[1] = trace;
        out[2] = lam > 0.0 ? trace / lam : 0.0;
        out[3] = (double)it;
    }
    cluster_sync();   // no CTA leaves while another may still write into it
}

}  // namespace tc
}  // namespace resbm
