// tc.cu -- host side of the sm_103a tensor-core kernels (tcgen05 + TMA) of the ResBM boundary.
//
// All tensor-core kernels are compiled in this one translation unit (they share the device
// error word of tc_common.cuh). Tensor maps are encoded per call through the driver entry point
// cuTensorMapEncodeTiled (no link-time dependency on libcuda).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <numeric>
#include <utility>

#include "tc.h"
#include "tc_common.cuh"
#include "tc_dec_fwd.cuh"
#include "tc_enc_fwd.cuh"
#include "tc_dec_bwd.cuh"
#include "tc_enc_bwd.cuh"
#include "tc_gemm.cuh"
#include "tc_spectral.cuh"
#include "tc_hbm_forms.cuh"

namespace resbm {

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// 2D bf16 (or fp32) tensor map over a row-major matrix (outer rows x inner columns, row pitch in bytes).
bool make_map(CUtensorMap *m, const void *ptr, uint64_t inner, uint64_t outer, uint64_t pitch_bytes,
              uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz,
              CUtensorMapDataType type = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16)
{
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {pitch_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t es[2] = {1, 1};
    return fn(m, type, 2, const_cast<void *>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

CUtensorMapSwizzle swizzle_for(uint32_t row_bytes)
{
    return row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
           : row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                             : CU_TENSOR_MAP_SWIZZLE_32B;
}

bool al16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Every kernel of this file is launched with programmatic stream serialization: it may be
// scheduled while the previous kernel of the stream is still finishing, and waits at its start
// (griddepcontrol.wait, before touching global memory) until that kernel has completed and its
// writes are visible. What overlaps is the launch itself and the placement of CTAs on SMs that
// the previous kernel has already left.
// `cluster` > 1 launches 1-D thread-block clusters of that many CTAs (the grid is a multiple).
template <typename... KArgs, typename... Args>
cudaError_t launch_clustered(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, int cluster,
                             cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args &&...args)
{
    return launch_clustered(kernel, grid, block, smem, 1, stream, std::forward<Args>(args)...);
}

// Dynamic shared memory attribute, set once per (kernel, device): `done` is the calling
// launcher's own per-device flag array (one per kernel instantiation).
constexpr int kMaxDev = 64;
template <typename K>
cudaError_t ensure_smem(K kernel, uint32_t bytes, int dev, std::atomic<uint8_t> (&done)[kMaxDev])
{
    if (dev >= 0 && dev < kMaxDev && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev >= 0 && dev < kMaxDev) done[dev].store(1, std::memory_order_release);
    return e;
}

// Number of clusters of `cl` CTAs of `kernel` (1-D, dynamic shared memory `smem`) that can be
// resident at once, asked once per (kernel, device, cluster size); `fit` is the calling
// launcher's own cache (count + 1; 0: not asked; index 0: 4 CTAs, 1: 2 CTAs). Needs the kernel's
// dynamic shared memory attribute set first. 0 if the query fails.
template <typename... KArgs>
int coresident_clusters(void (*kernel)(KArgs...), int cl, int threads, uint32_t smem, int dev,
                        std::atomic<int> (&fit)[kMaxDev][2])
{
    const int i = cl == 4 ? 0 : 1;
    const bool cached = dev >= 0 && dev < kMaxDev;
    int n = cached ? fit[dev][i].load(std::memory_order_acquire) - 1 : -1;
    if (n >= 0) return n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cl);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();   // not an error of the caller's stream: no clusters
        n = 0;
    }
    if (cached) fit[dev][i].store(n + 1, std::memory_order_release);
    return n;
}

// Grid and cluster size of a backward launch. The persistent grid would be g_full =
// min(128-token tiles, SMs) single CTAs; clusters of 4 are taken when at least 15/16 of g_full
// CTAs fit as co-resident clusters of 4 (the grid is then that many, a multiple of 4) and each
// CTA still gets at least `min_tokens` tokens, else clusters of 2 on the same terms, else single
// CTAs. Fewer, larger weight-gradient partials cost less than the few idle SMs (these kernels
// are bound by HBM, not by SM count), but the exchange has a cost per d chunk that only a long
// enough token range per CTA hides: min_tokens is the kernel's measured crossover.
struct BwdShape {
    int grid, cl;
};
// RESBM_CLUSTER=1, 2 or 4 forces that cluster size of the backward kernels (within the
// co-residency rule above, regardless of min_tokens), and 1 runs the encoder forward as single
// CTAs instead of pairs; unset or anything else: automatic. Read at every launch.
int forced_cluster()
{
    const char *v = getenv("RESBM_CLUSTER");
    if (!v) return 0;
    const int n = atoi(v);
    return n == 1 || n == 2 || n == 4 ? n : 0;
}
int bwd_full_grid(int64_t T, int sms)
{
    int64_t g = (T + 127) / 128;
    if (g > sms) g = sms;
    return (int)(g < 1 ? 1 : g);
}
int bwd_min_grid(int64_t T, int sms)
{
    const int gf = bwd_full_grid(T, sms);
    return (15 * gf + 15) / 16;
}
// RESBM_BWD_BALANCE=0 keeps the decoder backward's grid at the cluster rule's size; unset or
// anything else: balanced (bwd_balanced). Read at every launch.
bool bwd_balance_enabled()
{
    const char *v = getenv("RESBM_BWD_BALANCE");
    return !(v && v[0] == '0' && v[1] == 0);
}
// The fewest CTAs (a multiple of cl, at most g) that leave no CTA more whole tiles than g CTAs
// do: every CTA then has the same number of tiles or one fewer, as few as possible having
// fewer. At T = 65536 (512 tiles) on 144 CTAs, 80 CTAs make a fourth tile pass while 64 are
// done after three; 128 CTAs make the same four passes each, with fewer weight-gradient
// partial slots (32 clusters instead of 36). Measured at that size (bench, two A/B pairs): the
// decoder backward 116.5 -> 115.3 us; the encoder backward 211.0 -> 214.5 us (its epilogue's
// per-tile work gains from more SMs), so only the decoder backward takes it.
int bwd_balanced(int64_t T, int g, int cl)
{
    const int64_t U = (T + 127) / 128;
    const int64_t mt = (U + g - 1) / g;                    // the most tiles a CTA gets on g CTAs
    int64_t gb = (U + mt - 1) / mt;                        // the fewest CTAs with at most mt each
    gb = (gb + cl - 1) / cl * cl;
    return gb < g ? (int)gb : g;
}
template <typename... KArgs>
BwdShape bwd_shape(void (*kernel)(KArgs...), int64_t T, int sms, int threads, uint32_t smem, int clmax,
                   int64_t min_tokens, int dev, std::atomic<int> (&fit)[kMaxDev][2], bool balance)
{
    const int gf = bwd_full_grid(T, sms);
    const int forced = forced_cluster();
    const bool bal = balance && bwd_balance_enabled();
    for (int cl = 4; cl >= 2; cl /= 2) {
        if (cl > clmax || (forced && cl != forced)) continue;
        int64_t g = (int64_t)cl * coresident_clusters(kernel, cl, threads, smem, dev, fit);
        if (g > gf) g = gf;
        g -= g % cl;
        if (g >= cl && 16 * g >= 15 * (int64_t)gf && (forced || T >= min_tokens * g))
            return BwdShape{bal ? bwd_balanced(T, (int)g, cl) : (int)g, cl};
    }
    return BwdShape{bal ? bwd_balanced(T, gf, 1) : gf, 1};
}

bool tc_width_ok(int64_t m) { return m == 16 || m == 32 || m == 64 || m == 128; }

// NORM (k_dec_fwd): 0 Y; 1 Y and the row sums of squares into ss; 2 N = RMSNorm(Y) * gamma into Y
template <int M, int NORM = 0>
cudaError_t launch_dec_fwd(const resbm_desc &d, const void *B, const void *Wd1, const void *Wd2, void *Y,
                           const Ctx &c, float *ss = nullptr, const float *rstd = nullptr, const float *gamma32 = nullptr)
{
    using Cfg = tc::DecFwdCfg<M>;
    CUtensorMap m_wd2, m_y32, m_b;
    if (!make_map(&m_wd2, Wd2, d.d, d.m, d.d * 2, 64, M, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_y32, Y, d.d, d.T, d.d * 2, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_b, B, d.r, d.T, d.r * 2, Cfg::GB / 2, 128, swizzle_for(Cfg::GB)))
        return cudaErrorInvalidValue;
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_dec_fwd<M, NORM>, Cfg::SMEM_BYTES, c.device, smem_set);
    if (e != cudaSuccess) return e;
    tc::DecFwdArgs a{static_cast<const __nv_bfloat16 *>(Wd1), d.T, d.d, d.act, d.merge_identity,
                     ss, rstd, gamma32};
    // one CTA per SM, at most one per (tile, chunk) unit (the decoder forward splits tiles by columns)
    int64_t units = ((d.T + 127) / 128) * (d.d / Cfg::NCH);
    const int grid = (int)(units < c.sm_count ? (units < 1 ? 1 : units) : c.sm_count);
    e = launch(tc::k_dec_fwd<M, NORM>, grid, Cfg::THREADS, Cfg::SMEM_BYTES, c.stream, m_wd2, m_y32, m_b, a);
    count_launches(1);
    return e;
}

template <int M, bool REST>
cudaError_t launch_enc_fwd_t(const resbm_desc &d, const void *X, const void *F, const void *We1, const void *We2,
                             void *B, float *P, const Ctx &c)
{
    using Cfg = tc::EncFwdCfg<M>;
    const CUtensorMapSwizzle wswz = Cfg::WSW == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                                    : Cfg::WSW == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                     : CU_TENSOR_MAP_SWIZZLE_32B;
    tc::EncFwdMaps<REST> m;
    bool ok = make_map(&m.f128, F, d.d, d.T, d.d * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B) &&
              make_map(&m.we1, We1, d.m, d.d, d.m * 2, Cfg::WSW / 2, 64, wswz);
    if constexpr (REST)
        ok = ok && make_map(&m.frest, F, d.d, d.T, d.d * 2, 64, (uint32_t)(d.T % 128), CU_TENSOR_MAP_SWIZZLE_128B);
    if (!ok) return cudaErrorInvalidValue;
    auto kernel = tc::k_enc_fwd<M, REST>;
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(kernel, Cfg::SMEM_BYTES, c.device, smem_set);
    if (e != cudaSuccess) return e;
    tc::EncFwdArgs a{static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(We2),
                     static_cast<__nv_bfloat16 *>(B), P, d.T, d.d, d.act};
    // pairs of CTAs (clusters of 2), one pair per two SMs and at most one per tile, when there are
    // more tiles than SMs (single CTAs would make a second pass: the pairs split the tiles evenly)
    // and all the pairs fit at once; single CTAs otherwise (with at most one tile each they finish
    // together, and a pair's exchange of partial P costs more than its share of a tile saves:
    // T = 16384, d = 2048, 128 tiles: 22.3 us in pairs, 21.0 us single). RESBM_CLUSTER=1 forces
    // single CTAs, 2 or 4 pairs.
    const int64_t tiles = (d.T + 127) / 128;
    int cl = 1;
    int64_t grid = tiles < c.sm_count ? (tiles < 1 ? 1 : tiles) : c.sm_count;
    const int forced = forced_cluster();
    if (forced != 1 && (forced != 0 || tiles > c.sm_count)) {
        static std::atomic<int> fit[kMaxDev][2];
        int64_t pairs = tiles < c.sm_count / 2 ? (tiles < 1 ? 1 : tiles) : c.sm_count / 2;
        if (pairs >= 1 && coresident_clusters(kernel, 2, Cfg::THREADS, Cfg::SMEM_BYTES, c.device, fit) >= pairs) {
            cl = 2;
            grid = 2 * pairs;
        }
    }
    e = launch_clustered(kernel, (unsigned)grid, Cfg::THREADS, Cfg::SMEM_BYTES, cl, c.stream, m, a);
    count_launches(1);
    return e;
}
template <int M>
cudaError_t launch_enc_fwd(const resbm_desc &d, const void *X, const void *F, const void *We1, const void *We2,
                           void *B, float *P, const Ctx &c)
{
    return d.T % 128 ? launch_enc_fwd_t<M, true>(d, X, F, We1, We2, B, P, c) : launch_enc_fwd_t<M, false>(d, X, F, We1, We2, B, P, c);
}

// Scratch layout of the backward kernels: the d x m weight gradient has one fp32 slot per
// cluster (room for g_full single CTAs; tc_wgrad.cuh); the small one has one slot per (CTA, tile
// group). Every CTA has max_groups tile groups. The scratch size covers every grid the launch
// may pick (bwd_min_grid .. bwd_full_grid, and the balanced grids below them, which have no
// more tile groups per CTA and fewer CTAs), so it does not depend on the device's occupancy.
struct BwdPlan {
    int grid = 1, max_groups = 1, nch = 1;
    int64_t slots = 1;              // small partial slots
    float *part_big = nullptr;      // g_full x d x m
    float *part_small = nullptr;    // slots x small_elems
    size_t bytes = 0;
};

int bwd_max_groups(int64_t T, int grid, int nt)
{
    const int64_t U = (T + 127) / 128;   // tiles, split as token_range does
    const int64_t max_tiles = (U + grid - 1) / grid;
    const int64_t g = (max_tiles + nt - 1) / nt;
    return (int)(g < 1 ? 1 : g);
}

// grid > 0: the plan of that grid; grid == 0: the scratch size only (the largest over all grids).
BwdPlan bwd_plan(const resbm_desc &d, int sms, int grid, int nt, int64_t small_elems, void *ws)
{
    BwdPlan p;
    const int gf = bwd_full_grid(d.T, sms);
    int64_t small_slots = 0;
    if (grid > 0) {
        p.grid = grid;
        p.max_groups = bwd_max_groups(d.T, grid, nt);
        p.slots = (int64_t)grid * p.max_groups;
        small_slots = p.slots;
    } else {
        for (int g = bwd_min_grid(d.T, sms); g <= gf; ++g) {
            const int64_t s = (int64_t)g * bwd_max_groups(d.T, g, nt);
            if (s > small_slots) small_slots = s;
        }
    }
    p.nch = (int)(d.d / 128);
    WsCarver w(ws);
    p.part_big = w.take<float>((int64_t)gf * d.d * d.m);
    p.part_small = w.take<float>(small_slots * small_elems);
    p.bytes = w.used;
    return p;
}

// The two weight-gradient reductions of a backward op in one launch: the small (r x m) job
// first, on its own blocks, the large (d x m) one on the rest; one block per 32 float4 columns,
// the whole grid resident at once (8 blocks of 256 threads per SM).
const dim3 kReduceBlock(32, tc::kSlotGroups);
tc::ReduceJob reduce_job(const float *part, int64_t slots, int64_t rows, int64_t cols, float *out, int transpose,
                         int out4, int64_t cap)
{
    int64_t g = (rows * cols / 4 + 31) / 32;
    if (g > cap) g = cap;
    return tc::ReduceJob{part, slots, rows, cols, out, transpose, out4, (int)(g < 1 ? 1 : g), nullptr};
}
cudaError_t launch_reduce(const tc::ReduceJob &small, tc::ReduceJob big, const Ctx &c)
{
    const int64_t resident = (int64_t)c.sm_count * 8;
    const int64_t left = resident - small.blocks;
    if (big.blocks > left && left >= 1) big.blocks = (int)left;
    const cudaError_t e = launch(tc::k_reduce_slots, small.blocks + big.blocks, kReduceBlock, 0, c.stream, small, big);
    count_launches(1);
    return e;
}


template <int M>
cudaError_t launch_dec_bwd(const resbm_desc &d, const void *dY, const void *B, const void *Wd1, const void *Wd2,
                           void *dB, float *dWd1, float *dWd2, void *ws, const Ctx &c, bool after_independent)
{
    using Cfg = tc::DecBwdCfg<M>;
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_dec_bwd<M>, Cfg::SMEM_BYTES, c.device, smem_set);
    if (e != cudaSuccess) return e;
    static std::atomic<int> fit[kMaxDev][2];
    const BwdShape sh = bwd_shape(tc::k_dec_bwd<M>, d.T, c.sm_count, Cfg::THREADS, Cfg::SMEM_BYTES, Cfg::CLMAX,
                                  Cfg::CL_MIN_TOKENS, c.device, fit, true);
    const BwdPlan p = bwd_plan(d, c.sm_count, sh.grid, Cfg::NT, d.r * d.m, ws);
    CUtensorMap m_dy128, m_wd2, m_b, m_yr;
    if (!make_map(&m_dy128, dY, d.d, d.T, d.d * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_wd2, Wd2, d.d, d.m, d.d * 2, 64, M, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_b, B, d.r, d.T, d.r * 2, M, 128, swizzle_for(Cfg::RB)) ||
        !make_map(&m_yr, dY, d.d, d.T, d.d * 2, M, 128, swizzle_for(Cfg::RB)))
        return cudaErrorInvalidValue;
    tc::DecBwdArgs a{static_cast<const __nv_bfloat16 *>(Wd1),
                     static_cast<__nv_bfloat16 *>(dB),
                     tc::WgradArgs{p.part_big, p.nch},
                     p.part_small, d.T, d.d, d.act, d.merge_identity, p.max_groups, after_independent ? 1 : 0};
    e = launch_clustered(tc::k_dec_bwd<M>, p.grid, Cfg::THREADS, Cfg::SMEM_BYTES, sh.cl, c.stream, m_dy128,
                         m_wd2, m_b, m_yr, a);
    count_launches(1);
    if (e != cudaSuccess) return e;
    // dWd2 (m x d) = sum of the per-cluster slots (d x m), transposed; dWd1 (r x m) = sum of the slices
    const int64_t cap = (int64_t)c.sm_count * 8;
    return launch_reduce(reduce_job(p.part_small, p.slots, d.r, d.m, dWd1, 0, al16(dWd1), cap),
                         reduce_job(p.part_big, p.grid / sh.cl, d.d, d.m, dWd2, 1, 0, cap), c);
}

int dec_bwd_nt(int64_t m)
{
    return m <= 16 ? tc::DecBwdCfg<16>::NT : m <= 32 ? tc::DecBwdCfg<32>::NT : tc::DecBwdCfg<64>::NT;
}

// Scratch of the encoder backward: P (T x m fp32, used when the caller has none) and the slots.
struct EncBwdWs {
    float *P;
    BwdPlan plan;
    size_t bytes;
};

// grid > 0: the plan of that grid; grid == 0: the scratch size only (bwd_plan).
EncBwdWs enc_bwd_ws(const resbm_desc &d, int sms, int grid, void *ws)
{
    EncBwdWs w{};
    WsCarver c(ws);
    w.P = c.take<float>(d.T * d.m);
    char *rest = c.take<char>(0);
    const int nt = d.m <= 16 ? tc::EncBwdCfg<16>::NT : tc::EncBwdCfg<32>::NT;
    w.plan = bwd_plan(d, sms, grid, nt, d.m * d.r, ws ? rest : nullptr);
    w.bytes = c.used + w.plan.bytes;
    return w;
}

// P = F . We1 alone, by the kernel that the encoder forward takes for the shape, so that it matches a
// saved P bit for bit
cudaError_t recompute_P(const resbm_desc &d, const void *F, const void *We1, const void *We2, float *P, const Ctx &c);

template <int M>
cudaError_t launch_enc_bwd(const resbm_desc &d, const void *dB, const void *F, const float *P, const void *We1,
                           const void *We2, void *dF, void *dX, float *dWe1, float *dWe2, void *ws, const Ctx &c)
{
    using Cfg = tc::EncBwdCfg<M>;
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_enc_bwd<M>, Cfg::SMEM_BYTES, c.device, smem_set);
    if (e != cudaSuccess) return e;
    static std::atomic<int> fit[kMaxDev][2];
    const BwdShape sh = bwd_shape(tc::k_enc_bwd<M>, d.T, c.sm_count, Cfg::THREADS, Cfg::SMEM_BYTES, Cfg::CLMAX,
                                  Cfg::CL_MIN_TOKENS, c.device, fit, false);
    const EncBwdWs w = enc_bwd_ws(d, c.sm_count, sh.grid, ws);
    const BwdPlan &p = w.plan;
    CUtensorMap m_f128, m_we1, m_df32, m_db;
    if (!make_map(&m_f128, F, d.d, d.T, d.d * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_we1, We1, d.m, d.d, d.m * 2, M, 128, swizzle_for(Cfg::RB)) ||
        !make_map(&m_df32, dF, d.d, d.T, d.d * 2, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&m_db, dB, d.r, d.T, d.r * 2, M, 128, swizzle_for(Cfg::RB)))
        return cudaErrorInvalidValue;
    if (!P) {
        e = recompute_P(d, F, We1, We2, w.P, c);
        if (e != cudaSuccess) return e;
        P = w.P;
    }
    tc::EncBwdArgs a{P, static_cast<const __nv_bfloat16 *>(We2), static_cast<__nv_bfloat16 *>(dX),
                     tc::WgradArgs{p.part_big, p.nch}, p.part_small, d.T, d.d, d.act, p.max_groups};
    e = launch_clustered(tc::k_enc_bwd<M>, p.grid, Cfg::THREADS, Cfg::SMEM_BYTES, sh.cl, c.stream, m_f128, m_we1, m_df32, m_db, a);
    count_launches(1);
    if (e != cudaSuccess) return e;
    const int64_t cap = (int64_t)c.sm_count * 8;
    return launch_reduce(reduce_job(p.part_small, p.slots, d.m, d.r, dWe2, 0, al16(dWe2), cap),
                         reduce_job(p.part_big, p.grid / sh.cl, d.d, d.m, dWe1, 0, al16(dWe1), cap), c);
}

// ---- the GEMM chain (tc_gemm.cuh) --------------------------------------------------------
// C = A . B with A M x K (a_mn: stored K x M row-major, else M x K) and B K x N (b_mn: stored
// K x N row-major, else N x K), all bf16 with row pitches equal to the stored widths.
int gemm_bn(int64_t N) { return N > 128 ? 256 : 128; }

// The unit of a product: 128 rows on one CTA; 256 rows on one CTA (two 128-row MMAs sharing each B tile,
// GemmCfg's BM2); 256 rows on a CTA pair (two-CTA MMAs, k_gemm's PAIR).
enum GemmForm { kGemmSingle, kGemmBm2, kGemmPair };

char env_01(const char *name)
{
    const char *v = getenv(name);
    return v && (v[0] == '0' || v[0] == '1') && v[1] == 0 ? v[0] : 0;
}

// Pairs take every 256-column product with at least two row blocks. RESBM_GEMM_MC=0 turns them off, and
// RESBM_GEMM_BM2 = 0 / 1 never / always takes the one-CTA 256-row units where the shape allows (both read
// at every call: tuning and testing knobs). Without pairs the one-CTA 256-row units are for products
// without a lo half, where A is K-major, K (per split, for a weight gradient that may split it: wg) is
// long enough that a unit's epilogue, not overlapped with the next unit's products, is short next to
// them, and the units still give every SM one. Every form sums each output element over K in the same
// order; a weight gradient's split count can differ.
GemmForm gemm_form(int64_t M, int64_t N, int64_t K, bool lo, bool a_mn, int sms, bool wg)
{
    if (gemm_bn(N) != 256) return kGemmSingle;
    const char bm2 = env_01("RESBM_GEMM_BM2");
    if (bm2 == '1' && !lo) return kGemmBm2;
    if (M > 128 && env_01("RESBM_GEMM_MC") != '0') return kGemmPair;
    if (bm2 == '0' || lo || a_mn || M <= 256 || K < 2048) return kGemmSingle;
    int64_t units = ((M + 255) / 256) * ((N + 255) / 256);
    if (wg) units *= K / 2048 < 32 ? K / 2048 : 32;
    return units >= sms ? kGemmBm2 : kGemmSingle;
}

// Split-K of a product with few output tiles (the weight gradients, K = tokens): enough splits
// to give every SM (every pair of SMs) a unit, at most 32 and at least four 64-deep K slices per split.
int gemm_splits(int64_t M, int64_t N, int64_t K, int sms, GemmForm form = kGemmSingle)
{
    const int bn = gemm_bn(N), rows = form == kGemmSingle ? 128 : 256;
    const int64_t units = ((M + rows - 1) / rows) * ((N + bn - 1) / bn);
    const int64_t workers = form == kGemmPair ? sms / 2 : sms;
    if (4 * units >= 3 * workers) return 1;
    int64_t s = workers / units;
    // one-CTA 256-row units keep 2048 K per split (their epilogue is not overlapped with the next unit)
    const int64_t kmax = form == kGemmBm2 ? (K / 2048 > 1 ? K / 2048 : 1) : (K + 255) / 256;
    if (s > kmax) s = kmax;
    if (s > 32) s = 32;
    if (s < 1) s = 1;
    const int64_t kc = ((K + s - 1) / s + 63) / 64 * 64;
    return (int)((K + kc - 1) / kc);
}

// PAIR: CTA pairs (k_gemm); the grid is then two CTAs per co-resident pair, at most one pair per pair unit
// (returns cudaErrorNotSupported, before launching, when no pair
// fits: the caller runs single CTAs).
// TS: the outputs leave by TMA stores through `out` (k_gemm's TS forms; ENCP: F through out->o if it is
// stored); otherwise `out` is not read.
struct GemmOutMaps {
    CUtensorMap o, o2, lo;
};
template <int BN, bool AMN, bool BMN, bool ALO, bool ENCP = false, bool PAIR = false, bool BM2 = false, int TS = 0, bool RB = false>
cudaError_t launch_gemm_t(const CUtensorMap &ma, const CUtensorMap &malo, const CUtensorMap &mb,
                          tc::GemmShape g, const tc::GemmEp &ep, const Ctx &c, const GemmOutMaps *out = nullptr)
{
    using Cfg = tc::GemmCfg<BN, ALO, BM2, TS, PAIR, ENCP, RB, tc::gemm_halves(BN, AMN, ALO, ENCP, PAIR, BM2, TS)>;
    const GemmOutMaps none{ma, ma, ma};   // not read
    const GemmOutMaps &mo = out ? *out : none;
    auto kernel = tc::k_gemm<BN, AMN, BMN, ALO, ENCP, PAIR, BM2, TS, RB>;
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(kernel, Cfg::SMEM_BYTES, c.device, smem_set);
    if (e != cudaSuccess) return e;
    if (PAIR) {
        static std::atomic<int> fit[kMaxDev][2];
        const int pairs_fit = coresident_clusters(kernel, 2, Cfg::THREADS, Cfg::SMEM_BYTES, c.device, fit);
        const int64_t pair_units = (int64_t)((g.nm + 1) / 2) * g.nn * g.splits;
        const int64_t pairs = pair_units < pairs_fit ? pair_units : pairs_fit;
        if (pairs < 1) return cudaErrorNotSupported;
        g.turn = (int)(pairs / std::gcd<int64_t>(pairs, g.nn));
        e = launch_clustered(kernel, (unsigned)(2 * pairs), Cfg::THREADS, Cfg::SMEM_BYTES, 2, c.stream, ma, malo, mb, mo.o,
                             mo.o2, mo.lo, g, ep);
    } else {
        const int64_t grid = RB ? (g.M + g.rpc - 1) / g.rpc : g.units < c.sm_count ? g.units : c.sm_count;
        g.turn = (int)(grid / std::gcd<int64_t>(grid, g.nn));
        e = launch(kernel, (unsigned)grid, Cfg::THREADS, Cfg::SMEM_BYTES, c.stream, ma, malo, mb, mo.o, mo.o2, mo.lo, g, ep);
    }
    count_launches(1);
    return e;
}

// The TMA-store epilogue (k_gemm's TS form) unless RESBM_GEMM_TS=0 (read at every launch; a tuning
// and testing knob: both forms store the same bits).
bool ts_enabled()
{
    const char *v = getenv("RESBM_GEMM_TS");
    return !(v && v[0] == '0' && v[1] == 0);
}

// The TMA-store form of an epilogue and its output maps: 1 for one bf16 output (Y, dF, B, dB, the Newton-Schulz
// steps), 2 for the pre-activation and the activation's bf16 pair (P, A; Q, G; dQ; dP, A), or one fp32
// output (the weight gradients' slots), 0 for the rest, and for pointers or pitches TMA does not take.
int gemm_ts(const tc::GemmEp &ep, int64_t M, int64_t N, int splits, bool lo, GemmOutMaps *m)
{
    if (!ts_enabled()) return 0;
    bool ok = true;
    auto map = [&](CUtensorMap *t, const void *p, int64_t ld, bool f32, uint32_t cols, int64_t rows = 0) {
        const int64_t pitch = ld * (f32 ? 4 : 2);
        ok = ok && al16(p) && pitch % 16 == 0 &&
             make_map(t, p, N, rows ? rows : M, pitch, cols, 32, cols * (f32 ? 4 : 2) == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                      f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
    };
    switch (ep.mode) {
    case tc::GEP_BF16:
    case tc::GEP_ADD_AUX:
    case tc::GEP_DF:
    case tc::GEP_AXPBY:
        map(&m->o, ep.out, ep.ldo, false, 64);
        m->o2 = m->lo = m->o;
        return ok ? 1 : 0;
    case tc::GEP_F32:   // (split: one slot of M rows after the other, so the boxes of 32 rows may not cross M)
        if (ep.ldo != N || (splits > 1 && (M % 32 || ep.split_stride != M * N))) return 0;
        map(&m->o, ep.out, ep.ldo, true, 32, M * splits);
        m->o2 = m->lo = m->o;
        return ok ? 2 : 0;
    case tc::GEP_P_A:
    case tc::GEP_ACT:
    case tc::GEP_DACT: {
        if (lo || (ep.mode == tc::GEP_DACT && ep.lo && ep.out2 && N > 64)) return 0;   // (three: 64-column tiles only)
        const bool p_a = ep.mode == tc::GEP_P_A;
        const void *act = p_a ? ep.out2 : ep.out;   // the bf16 activation (or dQ, dP): always there
        map(p_a ? &m->o2 : &m->o, act, p_a ? ep.ldo2 : ep.ldo, false, 32);
        const CUtensorMap &a = p_a ? m->o2 : m->o;
        m->lo = a;
        if (ep.lo) map(&m->lo, ep.lo, p_a ? ep.ldo2 : ep.ldo, false, 32);
        CUtensorMap *other = p_a ? &m->o : &m->o2;   // P, Q (fp32) or A (bf16)
        const void *po = p_a ? ep.out : ep.out2;
        *other = a;
        if (po) map(other, po, p_a ? ep.ldo : ep.ldo2, ep.mode != tc::GEP_DACT, 32);
        return ok ? 2 : 0;
    }
    }
    return 0;
}

// The 64-deep K slices per piece of a sum (GemmShape::pc; launches without HALVES or PIECES do not read it), by the
// product alone, so that every form of it adds in the same order. Up to m = 64, where the chain can stand in for a
// fused kernel: a weight gradient's sum in pieces of 128 tokens, the least that a CTA of the fused decoder backward
// sums in one accumulator; P's and dQ's (K = d) in two halves. nk: slices per split. (Cost: the encoder forward by
// the chain 0.2 to 0.5 us of 10 to 20, the decoder backward 1 us of 50.)
int gemm_piece(int mode, bool wg, int64_t M, int64_t N, int64_t nk)
{
    if (wg) return (int)(M <= 64 && nk > 2 ? 2 : nk);
    const bool pre = mode == tc::GEP_F32 || mode == tc::GEP_P_A || mode == tc::GEP_ACT || mode == tc::GEP_DACT;
    return (int)(pre && N <= 64 && nk >= 4 ? (nk + 1) / 2 : nk);
}

// splits: 1 for every product whose epilogue is not a plain fp32 store; with splits > 1 the
// epilogue must be GEP_F32 into `splits` slots of M x N (ep.split_stride apart). A_lo: the lo
// half of A as a bf16 hi + lo pair (same shape and layout as A), or null. form: the unit as the
// caller chose it, or null to choose here.
cudaError_t gemm(const Ctx &c, int64_t M, int64_t N, int64_t K, const void *A, bool a_mn, const void *B, bool b_mn,
                 const tc::GemmEp &ep, int splits, const void *A_lo = nullptr, const GemmForm *form = nullptr)
{
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    const int bn = gemm_bn(N);
    CUtensorMap ma, malo, mbm;
    const bool okA = a_mn ? make_map(&ma, A, M, K, M * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)
                          : make_map(&ma, A, K, M, K * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    const bool okL = !A_lo ? true
                     : a_mn ? make_map(&malo, A_lo, M, K, M * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)
                            : make_map(&malo, A_lo, K, M, K * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    const bool lo = A_lo != nullptr;
    const GemmForm fm = form ? *form : gemm_form(M, N, K, lo, a_mn, c.sm_count, false);
    const bool bm2 = fm == kGemmBm2, pair = fm == kGemmPair;
    // K-major B: a pair's CTAs each load half of the B tile's rows
    const bool okB = b_mn ? make_map(&mbm, B, N, K, N * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)
                          : make_map(&mbm, B, K, N, K * 2, 64, (uint32_t)(pair ? bn / 2 : bn), CU_TENSOR_MAP_SWIZZLE_128B);
    if (!okA || !okL || !okB) return cudaErrorInvalidValue;
    if (!A_lo) malo = ma;   // not read
    tc::GemmShape g;
    g.M = M;
    g.N = N;
    g.K = K;
    g.splits = splits < 1 ? 1 : splits;
    g.kc = ((K + g.splits - 1) / g.splits + 63) / 64 * 64;
    g.splits = (int)((K + g.kc - 1) / g.kc);
    g.nm = (int)(bm2 ? (M + 255) / 256 : (M + 127) / 128);
    g.bnv = bn;
    if (pair && a_mn && b_mn && g.splits == 1) {
        // a weight gradient with about as many tiles as pairs: narrower tiles where that evens the last round out
        // (dWd2 of m = 512, d = 8192: 64 tiles of 256 columns on 76 pairs, 74 of 224)
        const int64_t m2 = (M + 255) / 256, pairs = c.sm_count / 2 > 0 ? c.sm_count / 2 : 1;
        int64_t best = 0;
        for (int w : {256, 224, 192, 160}) {
            const int64_t cost = (m2 * ((N + w - 1) / w) + pairs - 1) / pairs * w;
            if (best == 0 || cost < best) {
                best = cost;
                g.bnv = w;
            }
        }
    }
    g.nn = (int)((N + g.bnv - 1) / g.bnv);
    g.units = (int64_t)g.nm * g.nn * g.splits;
    if (g.units > INT32_MAX) return cudaErrorNotSupported;   // (2^38 rows, beyond any memory)
    g.rpc = 0;
    g.pc = gemm_piece(ep.mode, a_mn, M, N, (g.kc + 63) / 64);
    if (bm2) {
        if (!a_mn && b_mn) return launch_gemm_t<256, false, true, false, false, false, true>(ma, malo, mbm, g, ep, c);
        if (!a_mn && !b_mn) return launch_gemm_t<256, false, false, false, false, false, true>(ma, malo, mbm, g, ep, c);
        if (a_mn && b_mn) return launch_gemm_t<256, true, true, false, false, false, true>(ma, malo, mbm, g, ep, c);
        return cudaErrorNotSupported;
    }
    // TMA-store epilogues: on pairs, and for the products of up to 128 columns
    GemmOutMaps mo;
    // (an fp32 output on pairs only: beside the boxes the 128-column products keep 5 stages instead of 6, and
    // dWe1 of d = 8192, m = 128 went 84 -> 91 us)
    const bool ts_ok = ep.mode == tc::GEP_F32 ? pair && !lo : (pair || bn == 128) && !a_mn && g.splits == 1;
    const int ts = ts_ok ? gemm_ts(ep, M, N, g.splits, lo, &mo) : 0;
    if (ts == 2 && bn == 128) {   // P, dQ of m <= 128
        // 64-column tiles where N allows: A is what such a product reads, and beside the store boxes six stages of
        // it fit against five (N = 8, T = 12000, d = 3072 P 27.8 us by per-thread stores with six, 30.7 with five)
        const bool narrow = N <= 64;
        const int64_t rpc = (M + 32 * (int64_t)c.sm_count - 1) / (32 * (int64_t)c.sm_count) * 32;
        const bool rb = g.nm > c.sm_count && K >= 1024 && rpc < INT32_MAX;   // row-balanced units
        if (narrow && !b_mn && !make_map(&mbm, B, K, N, K * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;
        if (rb) {
            CUtensorMap mrest;
            if (!make_map(&mrest, A, K, M, K * 2, 64, rpc % 128 ? (uint32_t)(rpc % 128) : 128u, CU_TENSOR_MAP_SWIZZLE_128B))
                return cudaErrorInvalidValue;
            g.rpc = (int)rpc;
            if (narrow) return b_mn ? launch_gemm_t<64, false, true, false, false, false, false, 2, true>(ma, mrest, mbm, g, ep, c, &mo)
                                    : launch_gemm_t<64, false, false, false, false, false, false, 2, true>(ma, mrest, mbm, g, ep, c, &mo);
            return b_mn ? launch_gemm_t<128, false, true, false, false, false, false, 2, true>(ma, mrest, mbm, g, ep, c, &mo)
                        : launch_gemm_t<128, false, false, false, false, false, false, 2, true>(ma, mrest, mbm, g, ep, c, &mo);
        }
        if (narrow) return b_mn ? launch_gemm_t<64, false, true, false, false, false, false, 2>(ma, malo, mbm, g, ep, c, &mo)
                                : launch_gemm_t<64, false, false, false, false, false, false, 2>(ma, malo, mbm, g, ep, c, &mo);
        return b_mn ? launch_gemm_t<128, false, true, false, false, false, false, 2>(ma, malo, mbm, g, ep, c, &mo)
                    : launch_gemm_t<128, false, false, false, false, false, false, 2>(ma, malo, mbm, g, ep, c, &mo);
    }
    if (ts && bn == 128) {
        if (b_mn) return lo ? launch_gemm_t<128, false, true, true, false, false, false, 1>(ma, malo, mbm, g, ep, c, &mo)
                            : launch_gemm_t<128, false, true, false, false, false, false, 1>(ma, malo, mbm, g, ep, c, &mo);
        return lo ? launch_gemm_t<128, false, false, true, false, false, false, 1>(ma, malo, mbm, g, ep, c, &mo)
                  : launch_gemm_t<128, false, false, false, false, false, false, 1>(ma, malo, mbm, g, ep, c, &mo);
    }
    if (pair) {
        cudaError_t e = cudaErrorNotSupported;
        if (ts == 2 && a_mn) e = launch_gemm_t<256, true, true, false, false, true, false, 2>(ma, malo, mbm, g, ep, c, &mo);
        else if (ts == 2) e = b_mn ? launch_gemm_t<256, false, true, false, false, true, false, 2>(ma, malo, mbm, g, ep, c, &mo)
                                   : launch_gemm_t<256, false, false, false, false, true, false, 2>(ma, malo, mbm, g, ep, c, &mo);
        else if (ts && b_mn) e = lo ? launch_gemm_t<256, false, true, true, false, true, false, 1>(ma, malo, mbm, g, ep, c, &mo)
                                    : launch_gemm_t<256, false, true, false, false, true, false, 1>(ma, malo, mbm, g, ep, c, &mo);
        else if (ts) e = lo ? launch_gemm_t<256, false, false, true, false, true, false, 1>(ma, malo, mbm, g, ep, c, &mo)
                            : launch_gemm_t<256, false, false, false, false, true, false, 1>(ma, malo, mbm, g, ep, c, &mo);
        else if (!a_mn && b_mn) e = lo ? launch_gemm_t<256, false, true, true, false, true>(ma, malo, mbm, g, ep, c)
                                       : launch_gemm_t<256, false, true, false, false, true>(ma, malo, mbm, g, ep, c);
        else if (!a_mn && !b_mn) e = lo ? launch_gemm_t<256, false, false, true, false, true>(ma, malo, mbm, g, ep, c)
                                        : launch_gemm_t<256, false, false, false, false, true>(ma, malo, mbm, g, ep, c);
        else if (a_mn && b_mn) e = lo ? launch_gemm_t<256, true, true, true, false, true>(ma, malo, mbm, g, ep, c)
                                      : launch_gemm_t<256, true, true, false, false, true>(ma, malo, mbm, g, ep, c);
        if (e != cudaErrorNotSupported) return e;
        // no pair fits: whole tiles, and single CTAs need the whole-tile box for K-major B
        g.bnv = bn;
        g.nn = (int)((N + bn - 1) / bn);
        g.units = (int64_t)g.nm * g.nn * g.splits;
        if (!b_mn && !make_map(&mbm, B, K, N, K * 2, 64, (uint32_t)bn, CU_TENSOR_MAP_SWIZZLE_128B))
            return cudaErrorInvalidValue;
    }
    if (bn == 256) {
        if (!a_mn && b_mn) return lo ? launch_gemm_t<256, false, true, true>(ma, malo, mbm, g, ep, c)
                                     : launch_gemm_t<256, false, true, false>(ma, malo, mbm, g, ep, c);
        if (!a_mn && !b_mn) return lo ? launch_gemm_t<256, false, false, true>(ma, malo, mbm, g, ep, c)
                                      : launch_gemm_t<256, false, false, false>(ma, malo, mbm, g, ep, c);
        if (a_mn && b_mn) return lo ? launch_gemm_t<256, true, true, true>(ma, malo, mbm, g, ep, c)
                                    : launch_gemm_t<256, true, true, false>(ma, malo, mbm, g, ep, c);
    } else {
        if (!a_mn && b_mn) return lo ? launch_gemm_t<128, false, true, true>(ma, malo, mbm, g, ep, c)
                                     : launch_gemm_t<128, false, true, false>(ma, malo, mbm, g, ep, c);
        if (!a_mn && !b_mn) return lo ? launch_gemm_t<128, false, false, true>(ma, malo, mbm, g, ep, c)
                                      : launch_gemm_t<128, false, false, false>(ma, malo, mbm, g, ep, c);
        if (a_mn && b_mn) return lo ? launch_gemm_t<128, true, true, true>(ma, malo, mbm, g, ep, c)
                                    : launch_gemm_t<128, true, true, false>(ma, malo, mbm, g, ep, c);
    }
    return cudaErrorNotSupported;
}

tc::GemmEp ep_of(int mode, int act, void *out, int64_t ldo)
{
    tc::GemmEp e{};
    e.mode = mode;
    e.act = act;
    e.out = out;
    e.ldo = ldo;
    return e;
}

// A weight gradient W (M x N fp32) = A^T . B over K tokens (both operands MN-major), split over
// the tokens when it has few output tiles: the splits' fp32 slots go to `slots` and the job to
// sum them (in slot order) is returned in `job` (job->blocks = 0: nothing to reduce).
// A_lo: A as a bf16 hi + lo pair (or null). a_mn / b_mn: the operand majors (both MN-major for the
// weight gradients, whose K is the tokens).
// tr: W receives the transpose (N x M), by way of the slots (at least one) and the reduction; so does a W
// that is not 16-byte aligned.
cudaError_t wgrad(const Ctx &c, int64_t M, int64_t N, int64_t K, const void *A, const void *B, float *W, float *slots,
                  tc::ReduceJob *job, const void *A_lo = nullptr, bool a_mn = true, bool b_mn = true, bool tr = false)
{
    const GemmForm fm = gemm_form(M, N, K, A_lo != nullptr, a_mn, c.sm_count, true);
    const int s = gemm_splits(M, N, K, c.sm_count, fm);
    *job = tc::ReduceJob{};
    if (s <= 1 && !tr && al16(W)) return gemm(c, M, N, K, A, a_mn, B, b_mn, ep_of(tc::GEP_F32, 0, W, N), 1, A_lo, &fm);
    tc::GemmEp e = ep_of(tc::GEP_F32, 0, slots, N);
    e.split_stride = M * N;
    cudaError_t err = gemm(c, M, N, K, A, a_mn, B, b_mn, e, s, A_lo, &fm);
    if (err != cudaSuccess) return err;
    // the number of splits the launch took (gemm rounds K per split to 64)
    const int64_t kc = ((K + s - 1) / s + 63) / 64 * 64;
    const int64_t ns = (K + kc - 1) / kc;
    *job = reduce_job(slots, ns, M, N, W, tr, al16(W), (int64_t)c.sm_count * 8);
    return cudaSuccess;
}

cudaError_t reduce_jobs(const tc::ReduceJob &a, const tc::ReduceJob &b, const Ctx &c)
{
    if (a.blocks == 0 && b.blocks == 0) return cudaSuccess;
    const tc::ReduceJob none{};
    const tc::ReduceJob &first = a.blocks ? a : none;
    const tc::ReduceJob &second = a.blocks ? (b.blocks ? b : none) : b;
    const int blocks = first.blocks + second.blocks;
    const cudaError_t e = launch(tc::k_reduce_slots, blocks, kReduceBlock, 0, c.stream, first, second);
    count_launches(1);
    return e;
}

// Scratch of the GEMM chain of each op (grid == the device's SMs): the intermediate T x m
// tensors and the weight gradients' split slots.
struct GemmWs {
    float *P = nullptr, *Q = nullptr;
    __nv_bfloat16 *A = nullptr, *G = nullptr, *dQ = nullptr, *dP = nullptr;
    __nv_bfloat16 *A_lo = nullptr, *G_lo = nullptr, *dQ_lo = nullptr, *dP_lo = nullptr;   // remainders of hi + lo pairs
    float *slots1 = nullptr, *slots2 = nullptr;
    size_t bytes = 0;
};

// dF = dP . We1^T takes dP as a hi + lo pair up to this hidden width (K = m is short there and
// the product is bound by the dF stream; at larger m it would double the op's largest product)
constexpr int64_t kDfLoMaxM = 64;

size_t slot_floats(int64_t M, int64_t N, int64_t K, int sms)
{
    // room for every form (which one a launch takes can depend on the knobs)
    int s = 1;
    for (GemmForm f : {kGemmSingle, kGemmBm2, kGemmPair}) {
        const int n = gemm_splits(M, N, K, sms, f);
        if (n > s) s = n;
    }
    return s > 1 ? (size_t)(s * M * N) : 0;
}

// dWd1 = B^T . dQ takes dQ as a hi + lo pair (as dQ^T . B, transposed by its reduction) up to m = r = 64,
// where the chain runs in place of a fused kernel that does.
bool dwd1_pair(const resbm_desc &d) { return d.m == d.r && tc_width_ok(d.m) && d.m <= 64; }

GemmWs gemm_ws(const resbm_desc &d, int op, int sms, void *ws, bool have_P)
{
    GemmWs w;
    WsCarver cv(ws);
    const int64_t T = d.T, D = d.d, r = d.r, m = d.m;
    if (op == RESBM_OP_ENCODE_FWD) {
        w.A = cv.take<__nv_bfloat16>(T * m);
        w.A_lo = cv.take<__nv_bfloat16>(T * m);
    } else if (op == RESBM_OP_DECODE_FWD) {
        w.G = cv.take<__nv_bfloat16>(T * m);
    } else if (op == RESBM_OP_DECODE_BWD) {
        w.Q = cv.take<float>(T * m);
        w.G = cv.take<__nv_bfloat16>(T * m);
        w.G_lo = cv.take<__nv_bfloat16>(T * m);
        w.dQ = cv.take<__nv_bfloat16>(T * m);
        w.dQ_lo = cv.take<__nv_bfloat16>(T * m);
        w.slots1 = cv.take<float>(slot_floats(m, D, T, sms));   // dWd2
        const size_t s2 = slot_floats(r, m, T, sms);            // dWd1
        w.slots2 = cv.take<float>(dwd1_pair(d) && s2 < (size_t)(r * m) ? (size_t)(r * m) : s2);
    } else if (op == RESBM_OP_ENCODE_BWD) {
        if (!have_P) w.P = cv.take<float>(T * m);
        w.A = cv.take<__nv_bfloat16>(T * m);
        w.dP = cv.take<__nv_bfloat16>(T * m);
        if (m <= kDfLoMaxM) w.dP_lo = cv.take<__nv_bfloat16>(T * m);
        // dWe1, dWe2: at least one slot each, for gradients that are not 16-byte aligned
        const size_t s1 = slot_floats(D, m, T, sms), s2 = slot_floats(m, r, T, sms);
        w.slots1 = cv.take<float>(s1 ? s1 : (size_t)(D * m));
        w.slots2 = cv.take<float>(s2 ? s2 : (size_t)(m * r));
    }
    w.bytes = cv.used;
    return w;
}

}  // namespace

bool tc_supported(const resbm_desc &d, int op)
{
    if (d.dtype != RESBM_BF16 || d.m != d.r || !tc_width_ok(d.m)) return false;
    if (d.T > INT32_MAX || encode_fn() == nullptr) return false;
    if (op == RESBM_OP_DECODE_FWD) {
        const int64_t nch = d.m <= 32 ? 256 : 128;
        return d.d % nch == 0;
    }
    if (op == RESBM_OP_ENCODE_FWD) return d.m <= 64 && d.d % 64 == 0;
    if (op == RESBM_OP_DECODE_BWD) return d.m <= 64 && d.d % 128 == 0;
    if (op == RESBM_OP_ENCODE_BWD) return d.m <= 32 && d.d % 128 == 0;
    return false;
}

// Fused kernel or chain of products, where both take the shape. A CTA of a fused kernel streams whole
// 128-token tiles through all of d, so few tokens leave most SMs without work, and the backward kernels
// write one d x m partial gradient per CTA or cluster, which weighs against their one pass over the data
// when a CTA gets few tokens; the chain spreads both over the chip but reads the T x d input of a backward
// op twice and takes three to six launches (20 to 30 us at least). Measured, us, fused / chain (T x d):
// ("step": the boundary step with that op by the one or the other, whose other kernels leave their writes in L2)
//   encode fwd  m = 16: 256 x 2048 11 / 14, 1000 x 4096 18 / 19, 500 x 8192 30 / 30 (step 158 / 153), 4096 x 4096
//               17 / 20;  m = 32: 1000 x 512 12 / 9 (but step 39 / 40), 1000 x 1024 14 / 10, 1000 x 6144 29 / 24,
//               2000 x 1536 15 / 12, 2048 x 8192 32 / 29 (but step 227 / 240), 4096 x 1024 10.3 / 10.8, 16384 x
//               2048 18 / 22;  m = 64: 50000 x 2048 50 / 50 (but step 339 / 333), 65536 x 512 44 / 31, 65536 x
//               1024 48 / 42, 98304 x 768 61 / 53, 131072 x 1024 73 / 75 (but step 504 / 488), 65536 x 2048 60 / 64
//               (but step 419 / 414), 98304 x 2048 82 / 91 (step 576 / 577), 65536 x 4096 96 / 107 (step 653 / 658),
//               131072 x 2048 101 / 115 (step 719 / 726), 49152 x 4096 step 544 / 530, 65536 x 5120 step 798 / 800;
//               m = 128: 256 x 512 39 / 12 ... 65536 x 4096 155 / 121 (no fused kernel)
//   decode fwd  m = 64: 1000 x 4096 9 / 9, 65536 x 4096 83 / 102;  m = 128: 1000 x 512 17 / 11, 32768 x 8192
//               104 / 103, 65536 x 4096 121 / 115
//   decode bwd  m = 32: 1000 x 4096 39 / 34, 1000 x 8192 65 / 44, 4096 x 8192 77 / 54, 2048 x 4096 42 / 36 (but step
//               91 / 95), 6144 x 8192 79 / 70 (step 200 / 202), 16384 x 2048 30 / 46;  m = 64: 1000 x 512 21 / 30,
//               1000 x 4096 71 / 40, 16384 x 1920 50 / 55, 36864 x 1024 42 / 67, 39000 x 1536 122 / 92, 50000 x 1280
//               109 / 98, 76000 x 1024 99 / 123, 81920 x 1024 149 / 129, 262144 x 512 258 / 305;  steps: 19456 x 2048
//               184 / 178, 20000 x 4096 272 / 284, 30000 x 2048 220 / 243, 24576 x 8192 510 / 516, 38912 x 4096
//               426 / 435, 38912 x 6144 588 / 583, 45000 x 2048 366 / 324, 65536 x 4096 770 / 680
//   encode bwd  m = 16, steps: 1000 x 1408 50 / 54, 1000 x 2048 55 / 52, 4096 x 3072 79 / 77, 6000 x 4096 103 / 108,
//               8192 x 6144 149 / 153, 8192 x 8192 193 / 188;  m = 32, steps: 1 x 512 39 / 43, 1000 x 768 47 / 48,
//               1000 x 1024 52 / 51, 4096 x 2048 82 / 70, 12000 x 3072 132 / 137, 16384 x 4608 207 / 202, 20000 x
//               2048 140 / 142, 20000 x 3072 189 / 178, 32768 x 3072 238 / 235 (but alone 98 / 109), 32768 x 4096
//               301 / 290, 45000 x 4096 353 / 365;  m = 64: 256 x 512 26 / 20 ... 65536 x 4096 485 / 235 (no
//               fused kernel)
// One rule for an op alone and in a step, whose outputs are the ops' bit for bit. (Every entry on a device of 152 SMs:
// 19456 tokens give every CTA one whole tile there.)
// RESBM_CLUSTER set (the fused kernels' cluster size is being forced) keeps the fused kernels.
bool tc_preferred(const resbm_desc &d, int op, int sms)
{
    if (forced_cluster() || !gemm_supported(d, op)) return true;
    const int64_t round = 128 * (int64_t)sms;   // tokens: one whole tile per CTA
    switch (op) {
    case RESBM_OP_ENCODE_FWD:
        return d.m == 16   ? d.T > 1024 || d.d < 8192
               : d.m == 32 ? !(d.T <= 2048 && d.d >= 1024 && (d.T <= 1024 || d.d <= 2048))
                           : d.d >= 5120 ? 2 * d.T > 5 * round : d.d >= 2048 && d.T > 3 * round;
    case RESBM_OP_DECODE_FWD: return d.m <= 64;
    case RESBM_OP_DECODE_BWD:
        if (d.m == 16) return true;
        if (d.m == 32) return !(d.d >= 4096 && d.T <= d.d * 3 / 4 - 2048);
        if (d.d < 1024) return true;
        // (whole tiles a CTA: up to two; four, while the tensor is not much larger than L2; two of wide rows)
        if (d.d < 2048) return d.T <= 2 * round || (d.T > 3 * round && d.T * d.d <= (int64_t)76 << 20);
        return d.T > round && d.T <= 2 * round && d.T * d.d <= (int64_t)200 << 20;
    case RESBM_OP_ENCODE_BWD:
        if (d.m == 16) return d.d < 1024 + d.T / 2 || d.d < d.T * 3 / 4;
        if (d.T > 2 * round || d.d <= 768) return true;
        return d.T > round ? d.d <= 1024 + d.T / 16 : d.d < 512 + (d.T >= 8192 ? d.T / 4 : d.T / 5);
    }
    return true;
}

size_t tc_ws_bytes(const resbm_desc &d, int op, int sms)
{
    if (op == RESBM_OP_DECODE_BWD) return bwd_plan(d, sms, 0, dec_bwd_nt(d.m), d.r * d.m, nullptr).bytes;
    if (op == RESBM_OP_ENCODE_BWD) return enc_bwd_ws(d, sms, 0, nullptr).bytes;
    return 0;
}

cudaError_t tc_encode_fwd(const resbm_desc &d, const void *X, const void *F, const void *We1, const void *We2,
                          void *B, float *P, void *, const Ctx &c)
{
    if (!al16(X) || !al16(F) || !al16(We1) || !al16(We2) || !al16(B) || (P && !al16(P)))
        return cudaErrorNotSupported;
    switch (d.m) {
    case 16: return launch_enc_fwd<16>(d, X, F, We1, We2, B, P, c);
    case 32: return launch_enc_fwd<32>(d, X, F, We1, We2, B, P, c);
    case 64: return launch_enc_fwd<64>(d, X, F, We1, We2, B, P, c);
    }
    return cudaErrorNotSupported;
}

cudaError_t tc_decode_fwd(const resbm_desc &d, const void *B, const void *Wd1, const void *Wd2, void *Y, void *,
                          const Ctx &c)
{
    if (!al16(B) || !al16(Wd1) || !al16(Wd2) || !al16(Y)) return cudaErrorNotSupported;
    switch (d.m) {
    case 16: return launch_dec_fwd<16>(d, B, Wd1, Wd2, Y, c);
    case 32: return launch_dec_fwd<32>(d, B, Wd1, Wd2, Y, c);
    case 64: return launch_dec_fwd<64>(d, B, Wd1, Wd2, Y, c);
    }
    return cudaErrorNotSupported;
}

// gamma as fp32 (d), the row sums of squares (2 d / NCH slots of T), the T reciprocal RMS values
int rmsnorm_slots(const resbm_desc &d) { return (int)(2 * (d.d / (d.m <= 32 ? 256 : 128))); }   // NCH
size_t tc_rmsnorm_ws_bytes(const resbm_desc &d)
{
    return ((size_t)d.d + ((size_t)rmsnorm_slots(d) + 1) * (size_t)d.T) * sizeof(float);
}

template <int M>
cudaError_t dec_fwd_rmsnorm_t(const resbm_desc &d, const void *B, const void *Wd1, const void *Wd2,
                              const void *gamma, float eps, void *Y, void *N, float *ss, const Ctx &c)
{
    static_assert(tc::DecFwdCfg<M>::NCH == (M <= 32 ? 256 : 128), "rmsnorm_slots");
    const int ns = rmsnorm_slots(d);
    float *gamma32 = ss;   // first: d floats, a multiple of NCH, so the slots stay 16-byte aligned too
    ss += d.d;
    float *rstd = ss + (int64_t)ns * d.T;
    cudaError_t e = launch_dec_fwd<M, 1>(d, B, Wd1, Wd2, Y, c, ss);
    if (e != cudaSuccess) return e;
    const int64_t n = d.T > d.d ? d.T : d.d;
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)c.sm_count * 8) blocks = (int64_t)c.sm_count * 8;
    e = launch(tc::k_row_rstd, (unsigned)blocks, 256, 0, c.stream, (const float *)ss, ns, d.T, d.d, eps, rstd,
               static_cast<const __nv_bfloat16 *>(gamma), gamma32);
    count_launches(1);
    return e != cudaSuccess ? e : launch_dec_fwd<M, 2>(d, B, Wd1, Wd2, N, c, nullptr, rstd, gamma32);
}

cudaError_t tc_decode_fwd_rmsnorm(const resbm_desc &d, const void *B, const void *Wd1, const void *Wd2,
                                  const void *gamma, float eps, void *Y, void *N, void *ws, const Ctx &c)
{
    if (!al16(B) || !al16(Wd1) || !al16(Wd2) || !al16(Y) || !al16(N) || !al16(ws))
        return cudaErrorNotSupported;
    float *ss = static_cast<float *>(ws);
    switch (d.m) {
    case 16: return dec_fwd_rmsnorm_t<16>(d, B, Wd1, Wd2, gamma, eps, Y, N, ss, c);
    case 32: return dec_fwd_rmsnorm_t<32>(d, B, Wd1, Wd2, gamma, eps, Y, N, ss, c);
    case 64: return dec_fwd_rmsnorm_t<64>(d, B, Wd1, Wd2, gamma, eps, Y, N, ss, c);
    case 128: return dec_fwd_rmsnorm_t<128>(d, B, Wd1, Wd2, gamma, eps, Y, N, ss, c);
    }
    return cudaErrorNotSupported;
}

cudaError_t tc_decode_bwd(const resbm_desc &d, const void *dY, const void *B, const void *Wd1, const void *Wd2,
                          void *dB, float *dWd1, float *dWd2, void *ws, const Ctx &c, bool after_independent)
{
    if (!al16(dY) || !al16(B) || !al16(Wd1) || !al16(Wd2) || !al16(dB)) return cudaErrorNotSupported;
    switch (d.m) {
    case 16: return launch_dec_bwd<16>(d, dY, B, Wd1, Wd2, dB, dWd1, dWd2, ws, c, after_independent);
    case 32: return launch_dec_bwd<32>(d, dY, B, Wd1, Wd2, dB, dWd1, dWd2, ws, c, after_independent);
    case 64: return launch_dec_bwd<64>(d, dY, B, Wd1, Wd2, dB, dWd1, dWd2, ws, c, after_independent);
    }
    return cudaErrorNotSupported;
}

cudaError_t tc_encode_bwd(const resbm_desc &d, const void *dB, const void *F, const float *P, const void *We1,
                          const void *We2, void *dF, void *dX, float *dWe1, float *dWe2, void *ws, const Ctx &c)
{
    if (!al16(dB) || !al16(F) || (P && !al16(P)) || !al16(We1) || !al16(We2) || !al16(dF) || (dX && !al16(dX)))
        return cudaErrorNotSupported;
    switch (d.m) {
    case 16: return launch_enc_bwd<16>(d, dB, F, P, We1, We2, dF, dX, dWe1, dWe2, ws, c);
    case 32: return launch_enc_bwd<32>(d, dB, F, P, We1, We2, dF, dX, dWe1, dWe2, ws, c);
    }
    return cudaErrorNotSupported;
}

// ---- the GEMM chain of each op ------------------------------------------------------------
bool gemm_supported(const resbm_desc &d, int op)
{
    if (d.dtype != RESBM_BF16 || d.T > INT32_MAX || encode_fn() == nullptr) return false;
    if (d.d % 8 || d.r % 8 || d.m % 8) return false;   // 16-byte row pitches (TMA, vector epilogues)
    return op >= RESBM_OP_ENCODE_FWD && op <= RESBM_OP_ENCODE_BWD;
}

size_t gemm_ws_bytes(const resbm_desc &d, int op, int sms) { return gemm_ws(d, op, sms, nullptr, false).bytes; }

cudaError_t gemm_encode_fwd(const resbm_desc &d, const void *X, const void *F, const void *We1, const void *We2,
                            void *B, float *P, void *ws, const Ctx &c)
{
    if (!al16(X) || !al16(F) || !al16(We1) || !al16(We2) || !al16(B) || (P && !al16(P)) || !al16(ws))
        return cudaErrorNotSupported;
    const GemmWs w = gemm_ws(d, RESBM_OP_ENCODE_FWD, c.sm_count, ws, true);
    // P = F . We1 (saved if asked), A = phi(P)
    tc::GemmEp e1 = ep_of(tc::GEP_P_A, d.act, P, d.m);
    e1.out2 = w.A;
    e1.ldo2 = d.m;
    e1.lo = w.A_lo;
    cudaError_t e = gemm(c, d.T, d.m, d.d, F, false, We1, true, e1, 1);
    if (e != cudaSuccess) return e;
    // B = X[:, :r] + (A_hi + A_lo) . We2 (the truncating identity path added in the epilogue)
    tc::GemmEp e2 = ep_of(tc::GEP_ADD_AUX, d.act, B, d.r);
    e2.aux = X;
    e2.lda = d.d;
    e2.aux_cols = d.r;
    return gemm(c, d.T, d.r, d.m, w.A, false, We2, true, e2, 1, w.A_lo);
}

cudaError_t gemm_decode_fwd(const resbm_desc &d, const void *B, const void *Wd1, const void *Wd2, void *Y, void *ws,
                            const Ctx &c, bool keep_q)
{
    if (!al16(B) || !al16(Wd1) || !al16(Wd2) || !al16(Y) || !al16(ws)) return cudaErrorNotSupported;
    const GemmWs w = gemm_ws(d, keep_q ? RESBM_OP_DECODE_BWD : RESBM_OP_DECODE_FWD, c.sm_count, ws, true);
    // G = phi(B . Wd1); keep_q: with Q and G's remainder, where the decoder backward looks for them
    tc::GemmEp e1 = ep_of(tc::GEP_ACT, d.act, w.G, d.m);
    if (keep_q) {
        e1.out2 = w.Q;
        e1.ldo2 = d.m;
        e1.lo = w.G_lo;
    }
    cudaError_t e = gemm(c, d.T, d.m, d.r, B, false, Wd1, true, e1, 1);
    if (e != cudaSuccess) return e;
    // Y = G . Wd2 (+ B on the first r columns: the zero-padding identity path)
    tc::GemmEp e2 = ep_of(tc::GEP_ADD_AUX, d.act, Y, d.d);
    e2.aux = d.merge_identity ? B : nullptr;
    e2.lda = d.r;
    e2.aux_cols = d.merge_identity ? d.r : 0;
    return gemm(c, d.T, d.d, d.m, w.G, false, Wd2, true, e2, 1);
}

cudaError_t gemm_decode_bwd(const resbm_desc &d, const void *dY, const void *B, const void *Wd1, const void *Wd2,
                            void *dB, float *dWd1, float *dWd2, void *ws, const Ctx &c, bool have_q)
{
    if (!al16(dY) || !al16(B) || !al16(Wd1) || !al16(Wd2) || !al16(dB) || !al16(dWd1) || !al16(dWd2) || !al16(ws))
        return cudaErrorNotSupported;
    const GemmWs w = gemm_ws(d, RESBM_OP_DECODE_BWD, c.sm_count, ws, true);
    // Q = B . Wd1 (kept), G = phi(Q) as a hi + lo pair
    tc::GemmEp e1 = ep_of(tc::GEP_ACT, d.act, w.G, d.m);
    e1.out2 = w.Q;
    e1.ldo2 = d.m;
    e1.lo = w.G_lo;
    cudaError_t e = have_q ? cudaSuccess : gemm(c, d.T, d.m, d.r, B, false, Wd1, true, e1, 1);
    // dQ = (dY . Wd2^T) * phi'(Q)
    tc::GemmEp e2 = ep_of(tc::GEP_DACT, d.act, w.dQ, d.m);
    e2.aux = w.Q;
    e2.lda = d.m;
    e2.lo = w.dQ_lo;
    if (e == cudaSuccess) e = gemm(c, d.T, d.m, d.d, dY, false, Wd2, false, e2, 1);
    // dB = [merge] dY[:, :r] + (dQ_hi + dQ_lo) . Wd1^T
    tc::GemmEp e3 = ep_of(tc::GEP_ADD_AUX, d.act, dB, d.r);
    e3.aux = d.merge_identity ? dY : nullptr;
    e3.lda = d.d;
    e3.aux_cols = d.merge_identity ? d.r : 0;
    if (e == cudaSuccess) e = gemm(c, d.T, d.r, d.m, w.dQ, false, Wd1, false, e3, 1, w.dQ_lo);
    // dWd2 = (G_hi + G_lo)^T . dY, dWd1 = B^T . dQ (sums over the tokens; dQ as hi + lo up to m = r = 64)
    tc::ReduceJob j2, j1;
    if (e == cudaSuccess) e = wgrad(c, d.m, d.d, d.T, w.G, dY, dWd2, w.slots1, &j2, w.G_lo);
    if (e == cudaSuccess)
        e = dwd1_pair(d) ? wgrad(c, d.m, d.r, d.T, w.dQ, B, dWd1, w.slots2, &j1, w.dQ_lo, true, true, true)
                         : wgrad(c, d.r, d.m, d.T, B, w.dQ, dWd1, w.slots2, &j1);
    if (e == cudaSuccess) e = reduce_jobs(j1, j2, c);
    return e;
}

namespace {
cudaError_t recompute_P(const resbm_desc &d, const void *F, const void *We1, const void *We2, float *P, const Ctx &c)
{
    if (!(d.flags & RESBM_FLAG_GEMM) && tc_supported(d, RESBM_OP_ENCODE_FWD) && tc_preferred(d, RESBM_OP_ENCODE_FWD, c.sm_count) &&
        al16(We2))
        return d.m == 16   ? launch_enc_fwd<16>(d, nullptr, F, We1, We2, nullptr, P, c)
               : d.m == 32 ? launch_enc_fwd<32>(d, nullptr, F, We1, We2, nullptr, P, c)
                           : launch_enc_fwd<64>(d, nullptr, F, We1, We2, nullptr, P, c);
    return gemm(c, d.T, d.m, d.d, F, false, We1, true, ep_of(tc::GEP_F32, 0, P, d.m), 1);
}
}  // namespace

cudaError_t gemm_encode_bwd(const resbm_desc &d, const void *dB, const void *F, const float *P, const void *We1,
                            const void *We2, void *dF, void *dX, float *dWe1, float *dWe2, void *ws, const Ctx &c)
{
    if (!al16(dB) || !al16(F) || (P && !al16(P)) || !al16(We1) || !al16(We2) || !al16(dF) || (dX && !al16(dX)) || !al16(ws))
        return cudaErrorNotSupported;
    const GemmWs w = gemm_ws(d, RESBM_OP_ENCODE_BWD, c.sm_count, ws, P != nullptr);
    cudaError_t e = cudaSuccess;
    if (!P) {
        e = recompute_P(d, F, We1, We2, w.P, c);
        P = w.P;
    }
    // dP = (dB . We2^T) * phi'(P), and A = phi(P) for dWe2
    tc::GemmEp e1 = ep_of(tc::GEP_DACT, d.act, w.dP, d.m);
    e1.aux = P;
    e1.lda = d.m;
    e1.out2 = w.A;
    e1.ldo2 = d.m;
    e1.lo = w.dP_lo;
    if (e == cudaSuccess) e = gemm(c, d.T, d.m, d.r, dB, false, We2, false, e1, 1);
    // dF = dP . We1^T (dP as a hi + lo pair at small m), and dX[:, :r] += dB (the gradient of
    // the truncating identity path)
    tc::GemmEp e2 = ep_of(tc::GEP_DF, d.act, dF, d.d);
    e2.rmw = static_cast<__nv_bfloat16 *>(dX);
    e2.ldr = d.d;
    e2.aux = dB;
    e2.lda = d.r;
    e2.aux_cols = d.r;
    if (e == cudaSuccess) e = gemm(c, d.T, d.d, d.m, w.dP, false, We1, false, e2, 1, w.dP_lo);
    // dWe1 = F^T . dP, dWe2 = A^T . dB
    tc::ReduceJob j1, j2;
    if (e == cudaSuccess) e = wgrad(c, d.d, d.m, d.T, F, w.dP, dWe1, w.slots1, &j1);
    if (e == cudaSuccess) e = wgrad(c, d.m, d.r, d.T, w.A, dB, dWe2, w.slots2, &j2);
    if (e == cudaSuccess) e = reduce_jobs(j2, j1, c);
    return e;
}

// ---- the encoder fused into the FFN down-projection ---------------------------------------------
namespace {
int ffn_bn(int64_t d) { return d > 128 ? 256 : 128; }
int64_t ffn_slots(const resbm_desc &d) { return 2 * ((d.d + ffn_bn(d.d) - 1) / ffn_bn(d.d)); }
}  // namespace

bool ffn_encode_supported(const resbm_desc &d, int64_t f)
{
    return d.dtype == RESBM_BF16 && !(d.flags & RESBM_FLAG_LINEAR) && d.m % 8 == 0 && d.m <= 32 && d.r <= 32 &&
           d.d % 8 == 0 && f >= 1 && f % 8 == 0 && d.T <= INT32_MAX;
}

size_t ffn_encode_ws_bytes(const resbm_desc &d, int64_t f)
{
    (void)f;
    WsCarver cv(nullptr);
    cv.take<float>(ffn_slots(d) * d.T * d.m);
    return cv.used;
}

cudaError_t tc_ffn_down_encode(const resbm_desc &d, int64_t f, const void *H, const void *W2, const void *X,
                               const void *We1, const void *We2, void *B, float *P, void *F_out, void *ws,
                               const Ctx &c)
{
    if (!al16(H) || !al16(W2) || !al16(We1) || !al16(ws) || (F_out && !al16(F_out)) || (P && !al16(P)) ||
        encode_fn() == nullptr)
        return cudaErrorNotSupported;
    const int bn = ffn_bn(d.d);
    CUtensorMap ma, mb;
    if (!make_map(&ma, H, f, d.T, f * 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&mb, W2, d.d, f, d.d * 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    tc::GemmShape g{};
    g.M = d.T;
    g.N = d.d;
    g.K = f;
    g.splits = 1;
    g.kc = (f + 63) / 64 * 64;
    g.nm = (int)((d.T + 127) / 128);
    g.nn = (int)((d.d + bn - 1) / bn);
    g.bnv = bn;
    g.units = (int64_t)g.nm * g.nn;
    tc::GemmEp e{};
    e.out = F_out;
    e.ldo = d.d;
    e.we1 = static_cast<const __nv_bfloat16 *>(We1);
    e.pslots = static_cast<float *>(ws);
    e.slot_stride = d.T * d.m;
    e.pm = (int)d.m;
    GemmOutMaps mo{ma, ma, ma};
    if (F_out && !make_map(&mo.o, F_out, d.d, d.T, d.d * 2, 64, 32, CU_TENSOR_MAP_SWIZZLE_128B)) return cudaErrorInvalidValue;
    cudaError_t err = cudaErrorNotSupported;
    // (lo: never in one-CTA 256-row units: measured 0.31 -> 0.47 ms at T = 16384, f = 5632, d = 2048, the
    // P partials' epilogue no longer hidden behind the next unit's products)
    if (gemm_form(d.T, d.d, f, true, false, c.sm_count, false) == kGemmPair) err = launch_gemm_t<256, false, true, false, true, true>(ma, ma, mb, g, e, c, &mo);
    if (err == cudaErrorNotSupported)
        err = bn == 256 ? launch_gemm_t<256, false, true, false, true>(ma, ma, mb, g, e, c, &mo)
                        : launch_gemm_t<128, false, true, false, true>(ma, ma, mb, g, e, c, &mo);
    if (err != cudaSuccess) return err;
    err = launch(tc::k_enc_finish, (unsigned)((d.T + 7) / 8), 256, 0, c.stream, (const float *)ws,
                 (int)ffn_slots(d), d.T * d.m, d.T, (int)d.m, (int)d.r, d.act, P,
                 static_cast<const __nv_bfloat16 *>(We2), static_cast<const __nv_bfloat16 *>(X), d.d,
                 static_cast<__nv_bfloat16 *>(B));
    count_launches(1);
    return err;
}

// ---- Muon's Newton-Schulz orthogonalisation and the effective rank ----------------------------
namespace {
// Scratch: the sum-of-squares partials, the two bf16 iterates (or the Gram matrix and its split
// slots for the effective rank), and the s x s products (s = min(rows, cols)).
struct MatrixWs {
    double *part = nullptr;
    __nv_bfloat16 *X = nullptr, *A = nullptr, *Bm = nullptr;
    float *gram = nullptr, *slots = nullptr;
    double *out = nullptr;
    size_t bytes = 0;
};
MatrixWs matrix_ws(int op, int64_t rows, int64_t cols, int sms, void *ws)
{
    MatrixWs w;
    WsCarver cv(ws);
    const int64_t sd = rows < cols ? rows : cols, ld = rows < cols ? cols : rows;
    if (op == RESBM_OP_NEWTON_SCHULZ) {
        w.part = cv.take<double>(tc::kSqBlocks);
        w.X = cv.take<__nv_bfloat16>(rows * cols);
        w.A = cv.take<__nv_bfloat16>(sd * sd);
        w.Bm = cv.take<__nv_bfloat16>(sd * sd);
        if (ld >= 2048) w.slots = cv.take<float>(slot_floats(sd, sd, ld, sms));   // (shorter: one launch is quicker)
        if (slot_floats(sd, sd, ld, sms) == 0) w.slots = nullptr;
    } else {
        w.gram = cv.take<float>(sd * sd);
        w.slots = cv.take<float>(slot_floats(sd, sd, ld, sms));
    }
    w.bytes = cv.used;
    return w;
}
}  // namespace

namespace {
template <int SDP, typename TG>
cudaError_t launch_ns_t(int64_t rows, int64_t cols, const void *G, int steps, const float coef[3], float eps, void *out,
                        const Ctx &c)
{
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_newton_schulz<SDP, TG>, tc::kNsMaxSmem, c.device, smem_set);
    if (e != cudaSuccess) return e;
    const bool tall = rows > cols;
    const int64_t sd = tall ? cols : rows, ld = tall ? rows : cols;
    const tc::NsLayout l = tc::ns_layout(SDP, ld);
    e = launch_clustered(tc::k_newton_schulz<SDP, TG>, l.cl, tc::kNsThreads, l.bytes, l.cl, c.stream,
                         static_cast<const TG *>(G), (int)sd, ld, tall ? 1 : 0, steps, coef[0], coef[1], coef[2], eps,
                         static_cast<__nv_bfloat16 *>(out));
    count_launches(1);
    return e;
}
template <typename TG>
cudaError_t launch_ns(int64_t rows, int64_t cols, const void *G, int steps, const float coef[3], float eps, void *out,
                      const Ctx &c)
{
    switch (tc::ns_sdp(rows < cols ? rows : cols)) {
    case 16: return launch_ns_t<16, TG>(rows, cols, G, steps, coef, eps, out, c);
    case 32: return launch_ns_t<32, TG>(rows, cols, G, steps, coef, eps, out, c);
    case 48: return launch_ns_t<48, TG>(rows, cols, G, steps, coef, eps, out, c);
    default: return launch_ns_t<64, TG>(rows, cols, G, steps, coef, eps, out, c);
    }
}
}  // namespace

size_t matrix_ws_bytes(int op, int64_t rows, int64_t cols, int sms) { return matrix_ws(op, rows, cols, sms, nullptr).bytes; }

bool matrix_supported(int64_t rows, int64_t cols)
{
    return rows >= 1 && cols >= 1 && rows % 8 == 0 && cols % 8 == 0 && rows <= INT32_MAX && cols <= INT32_MAX;
}

cudaError_t tc_newton_schulz(int64_t rows, int64_t cols, const void *G, bool g_f32, int steps, const float coef[3],
                             float eps, void *X_out, void *ws, const Ctx &c)
{
    if (!al16(G) || !al16(X_out) || !al16(ws) || encode_fn() == nullptr) return cudaErrorNotSupported;
    // a small side of up to 64 whose columns fit in a cluster's shared memory: one launch
    if (tc::ns_fused_ok(rows, cols))
        return g_f32 ? launch_ns<float>(rows, cols, G, steps, coef, eps, X_out, c)
                     : launch_ns<__nv_bfloat16>(rows, cols, G, steps, coef, eps, X_out, c);
    const MatrixWs w = matrix_ws(RESBM_OP_NEWTON_SCHULZ, rows, cols, c.sm_count, ws);
    const int64_t n = rows * cols;
    __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(X_out);
    // the iterates alternate between the output and the scratch copy so that the last one lands in
    // the output: X0 in the scratch copy for an odd number of steps
    __nv_bfloat16 *cur = steps % 2 ? w.X : out, *nxt = steps % 2 ? out : w.X;
    int64_t grid = (n + 255) / 256;
    if (grid > (int64_t)c.sm_count * 8) grid = (int64_t)c.sm_count * 8;
    cudaError_t e;
    if (g_f32) {
        e = launch(tc::k_sumsq<float>, tc::kSqBlocks, 256, 0, c.stream, static_cast<const float *>(G), n, w.part);
        if (e == cudaSuccess)
            e = launch(tc::k_scale_bf16<float>, (unsigned)grid, 256, 0, c.stream, static_cast<const float *>(G), n,
                       (const double *)w.part, eps, cur);
    } else {
        e = launch(tc::k_sumsq<__nv_bfloat16>, tc::kSqBlocks, 256, 0, c.stream, static_cast<const __nv_bfloat16 *>(G),
                   n, w.part);
        if (e == cudaSuccess)
            e = launch(tc::k_scale_bf16<__nv_bfloat16>, (unsigned)grid, 256, 0, c.stream,
                       static_cast<const __nv_bfloat16 *>(G), n, (const double *)w.part, eps, cur);
    }
    count_launches(2);
    const bool wide = rows <= cols;
    const int64_t sd = wide ? rows : cols;
    for (int k = 0; k < steps && e == cudaSuccess; ++k) {
        // A = X X^T (wide) or X^T X (tall): the s x s Gram matrix of the iterate
        // (split over the long side where it has few tiles: 512 x 512 from 8192 columns took four pairs 42 us)
        tc::ReduceJob job{};
        if (w.slots) {
            e = wgrad(c, sd, sd, wide ? cols : rows, cur, cur, nullptr, w.slots, &job, nullptr, !wide, !wide, true);
            job.transpose = 0;   // (wgrad's way by the slots; the Gram matrix is stored as it is)
            job.out_bf16 = w.A;
            if (e == cudaSuccess) e = reduce_jobs(job, tc::ReduceJob{}, c);
        } else {
            e = wide ? gemm(c, sd, sd, cols, cur, false, cur, false, ep_of(tc::GEP_BF16, 0, w.A, sd), 1)
                     : gemm(c, sd, sd, rows, cur, true, cur, true, ep_of(tc::GEP_BF16, 0, w.A, sd), 1);
        }
        // Bm = b A + c A A
        tc::GemmEp eb = ep_of(tc::GEP_AXPBY, 0, w.Bm, sd);
        eb.aux = w.A;
        eb.lda = eb.aux_cols = sd;
        eb.alpha = coef[2];
        eb.beta = coef[1];
        if (e == cudaSuccess) e = gemm(c, sd, sd, sd, w.A, false, w.A, true, eb, 1);
        // X <- a X + Bm X (wide) or a X + X Bm (tall; Bm is symmetric)
        tc::GemmEp ex = ep_of(tc::GEP_AXPBY, 0, nxt, cols);
        ex.aux = cur;
        ex.lda = ex.aux_cols = cols;
        ex.alpha = 1.0f;
        ex.beta = coef[0];
        if (e == cudaSuccess)
            e = wide ? gemm(c, rows, cols, rows, w.Bm, false, cur, true, ex, 1)
                     : gemm(c, rows, cols, cols, cur, false, w.Bm, true, ex, 1);
        __nv_bfloat16 *t = cur;
        cur = nxt;
        nxt = t;
    }
    return e;
}

cudaError_t tc_effective_rank(int64_t rows, int64_t cols, const void *W, double *out, void *ws, const Ctx &c)
{
    if (!al16(W) || !al16(ws) || encode_fn() == nullptr) return cudaErrorNotSupported;
    const MatrixWs w = matrix_ws(RESBM_OP_EFFECTIVE_RANK, rows, cols, c.sm_count, ws);
    const bool tall = rows >= cols;
    const int64_t sd = tall ? cols : rows, ld = tall ? rows : cols;
    if (sd > tc::kPowMaxN) return cudaErrorNotSupported;
    // the Gram matrix of the smaller side: W^T W (tall) or W W^T (wide), fp32 sums of bf16 products
    tc::ReduceJob job;
    cudaError_t e = tall ? wgrad(c, sd, sd, ld, W, W, w.gram, w.slots, &job)
                         : wgrad(c, sd, sd, ld, W, W, w.gram, w.slots, &job, nullptr, false, false);
    if (e == cudaSuccess) e = reduce_jobs(job, tc::ReduceJob{}, c);
    if (e == cudaSuccess) {
        const bool small = sd <= tc::kLzSmallN;
        auto kernel = small ? tc::k_lanczos_small : tc::k_lanczos_top;
        const uint32_t smem = 4u * (uint32_t)(small ? tc::lanczos_small((int)sd).floats : tc::lanczos_layout((int)sd).floats);
        static std::atomic<uint8_t> set_small[kMaxDev], set_top[kMaxDev];
        e = ensure_smem(kernel, tc::kLzMaxSmem, c.device, small ? set_small : set_top);
        if (e != cudaSuccess) return e;
        e = launch_clustered(kernel, tc::kLzCl, tc::kLzThreads, smem, tc::kLzCl, c.stream, (const float *)w.gram, (int)sd,
                             20000, 1e-5f, out);
        count_launches(1);
    }
    return e;
}

namespace tc {
// One thread waits on an mbarrier that nothing arrives on; mbar_wait gives up after kWaitNs,
// sets the timeout bit of the error word and returns, and the kernel exits normally.
__global__ void k_wait_selftest()
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(smem_u32(&bar), 0);
}
}  // namespace tc

namespace {
// The 3-D view of the 3-D load form: {64 columns, rows, 64 column blocks} with the blocks 128
// bytes apart, so that one box {64, 128, 2} holds two neighbouring 64-column blocks of 128 rows
// and lands as two 64 x 128 swizzled boxes.
bool make_map_form3d(CUtensorMap *m, const void *ptr, uint64_t rows)
{
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {64, rows, (cuuint64_t)tc::kFormBlocks};
    cuuint64_t strides[2] = {(cuuint64_t)tc::kFormBlocks * 128, 128};
    cuuint32_t box[3] = {64, 128, 2};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int FORM>
cudaError_t launch_form_load(const CUtensorMap &m, const void *a, int64_t boxes, const Ctx &c)
{
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_form_load<FORM>, tc::kFormSmem, c.device, smem_set);
    if (e != cudaSuccess) return e;
    tc::k_form_load<FORM><<<c.sm_count, 128, tc::kFormSmem, c.stream>>>(m, static_cast<const uint8_t *>(a), boxes);
    return cudaGetLastError();
}

template <int FORM>
cudaError_t launch_form_store(const CUtensorMap &m, void *b, int64_t boxes, const Ctx &c)
{
    static std::atomic<uint8_t> smem_set[kMaxDev];
    cudaError_t e = ensure_smem(tc::k_form_store<FORM>, tc::kFormSmem, c.device, smem_set);
    if (e != cudaSuccess) return e;
    tc::k_form_store<FORM><<<c.sm_count, 128, tc::kFormSmem, c.stream>>>(m, static_cast<uint8_t *>(b), boxes);
    return cudaGetLastError();
}
}  // namespace

cudaError_t tc_hbm_form(int form, const void *a, void *b, int64_t bytes, const Ctx &c)
{
    const int64_t boxes = bytes / tc::kFormBox, rows = bytes / (tc::kFormBlocks * 128), n16 = bytes / 16;
    const int vgrid = c.sm_count * 4;
    CUtensorMap m;
    std::memset(&m, 0, sizeof(m));
    const bool reads = form == RESBM_HBM_READ_TMA_2D || form == RESBM_HBM_READ_TMA_2D_PAIR ||
                       form == RESBM_HBM_READ_TMA_2D_TILES;
    const bool writes = form == RESBM_HBM_WRITE_TMA_2D || form == RESBM_HBM_WRITE_TMA_2D_TILES;
    if ((reads || writes) && !make_map(&m, reads ? a : b, tc::kFormBlocks * 64, (uint64_t)rows,
                                       tc::kFormBlocks * 128, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (form == RESBM_HBM_READ_TMA_3D && !make_map_form3d(&m, a, (uint64_t)rows)) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    switch (form) {
    case RESBM_HBM_READ_V4:
        tc::k_form_read_v4<<<vgrid, 512, 0, c.stream>>>(static_cast<const uint4 *>(a), n16, static_cast<unsigned *>(b));
        e = cudaGetLastError();
        break;
    case RESBM_HBM_WRITE_V4:
        tc::k_form_write_v4<<<vgrid, 512, 0, c.stream>>>(static_cast<uint4 *>(b), n16);
        e = cudaGetLastError();
        break;
    case RESBM_HBM_COPY_V4:
        tc::k_form_copy_v4<<<vgrid, 512, 0, c.stream>>>(static_cast<const uint4 *>(a), static_cast<uint4 *>(b), n16);
        e = cudaGetLastError();
        break;
    case RESBM_HBM_READ_TMA_2D: e = launch_form_load<tc::kLoad2d>(m, a, boxes, c); break;
    case RESBM_HBM_READ_TMA_2D_PAIR: e = launch_form_load<tc::kLoad2dPair>(m, a, boxes, c); break;
    case RESBM_HBM_READ_TMA_3D: e = launch_form_load<tc::kLoad3d>(m, a, boxes, c); break;
    case RESBM_HBM_READ_BULK: e = launch_form_load<tc::kLoadBulk>(m, a, boxes, c); break;
    case RESBM_HBM_WRITE_TMA_2D: e = launch_form_store<tc::kStore2d>(m, b, boxes, c); break;
    case RESBM_HBM_WRITE_BULK: e = launch_form_store<tc::kStoreBulk>(m, b, boxes, c); break;
    case RESBM_HBM_READ_TMA_2D_TILES: e = launch_form_load<tc::kLoadTiles>(m, a, boxes, c); break;
    case RESBM_HBM_WRITE_TMA_2D_TILES: e = launch_form_store<tc::kStoreTiles>(m, b, boxes, c); break;
    default: return cudaErrorInvalidValue;
    }
    count_launches(1);
    return e;
}

cudaError_t tc_wait_selftest(const Ctx &c)
{
    tc::k_wait_selftest<<<1, 32, 0, c.stream>>>();
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t tc_device_error(unsigned int *code, bool clear)
{
    cudaError_t e = cudaMemcpyFromSymbol(code, tc::g_resbm_device_error, sizeof(unsigned int));
    if (e == cudaSuccess && clear && *code) {
        const unsigned int zero = 0;
        e = cudaMemcpyToSymbol(tc::g_resbm_device_error, &zero, sizeof(zero));
    }
    return e;
}

}  // namespace resbm
