// libsbn: the C ABI declared in include/sbn.h.  Host side only validates arguments, encodes TMA
// tensor maps and enqueues kernels on the caller's stream; every step of the path runs in the
// kernels of this translation unit.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <vector>

#include "sbn.h"
#include "sbn_common.cuh"
#include "quant_act.cuh"
#include "norm_quant_act.cuh"
#include "quantize_mask_pack.cuh"
#include "quantize_mask_pack_stream.cuh"
#include "canonical_layout.cuh"
#include "gemm_tcgen05.cuh"
#include "quant_rows.cuh"
#include "gemm_pair_tcgen05.cuh"
#include "gemm_splitk_cluster_tcgen05.cuh"
#include "gemm_splitk_wide_tcgen05.cuh"
#include "gemm_packed_cluster_tcgen05.cuh"
#include "gemm_fused_act_cluster_tcgen05.cuh"
#include "gemm_few_tokens_mma.cuh"
#include "backward_prep.cuh"
#include "gemm_bf16_pair_tcgen05.cuh"

namespace sbn {

// ------------------------------------------------------------------------------------------------
// host state
// ------------------------------------------------------------------------------------------------
static int g_force_token_tile = 0;
static int g_force_split_k = 0;            // > 0: global-atomics split-K factor; < 0: cluster split-K of that size

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            fn = reinterpret_cast<EncodeTiledFn>(p);
        }
    });
    return fn;
}

// 3-D view [d2][d1][1 KB] of tiled operand data (1 KB rows of 128 x uint64); box {1 KB, b1, b2}.
static bool encode_3d_1k(CUtensorMap* map, const void* base, uint64_t d1, uint64_t d2, uint32_t b1, uint32_t b2) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn || b1 == 0 || b1 > 256 || b2 == 0 || b2 > 256) return false;
    cuuint64_t dims[3] = {128, d1, d2};
    cuuint64_t strides[2] = {1024, 1024 * d1};
    cuuint32_t box[3] = {128, b1, b2};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<void*>(base), dims, strides, box,
                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// 2-D row-major output tensor y [T][N] (fp32 or bf16) with a 32-feature x box_tokens box.
static bool encode_2d_out(CUtensorMap* map, const void* base, uint64_t N, uint64_t T, bool bf16,
                          uint32_t box_tokens, uint32_t box_features = 32) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const uint64_t es = bf16 ? 2 : 4;
    cuuint64_t dims[2] = {N, T};
    cuuint64_t strides[1] = {N * es};
    cuuint32_t box[2] = {box_features, box_tokens};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                    const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Flat array of tiled operand data viewed as rows of 1 KB (128 x uint64); box = box_rows rows.
static bool encode_flat_1k(CUtensorMap* map, const void* base, uint64_t total_bytes, uint32_t box_rows) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn || total_bytes % 1024 != 0) return false;
    cuuint64_t dims[2] = {128, total_bytes / 1024};
    cuuint64_t strides[1] = {1024};
    cuuint32_t box[2] = {128, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(base), dims, strides, box,
                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Row-major bf16 matrix [rows][ld] of which `inner` columns are valid, fetched in boxes of 64 columns x
// box_rows rows with the 128-byte swizzle: the box lands in shared memory as the K-major operand image.
static bool encode_2d_bf16_sw128(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint64_t ld, uint32_t box_rows) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn || box_rows == 0 || box_rows > 256 || (ld * 2) % 16 != 0) return false;
    cuuint64_t dims[2] = {inner, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Row-major bf16 matrix [rows][cols], cols % 64 == 0, fetched as `blocks` blocks of 64 columns x 64 rows, block by block.
static bool encode_3d_bf16_blocks(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, uint32_t blocks) {
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {64, rows, cols / 64};
    cuuint64_t strides[2] = {cols * 2, 128};
    cuuint32_t box[3] = {64, 64, blocks};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

static inline bool misaligned(const void* p, size_t a) {
    return (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0;
}

static inline int pick_token_tile(int T) {
    if (g_force_token_tile == 64 || g_force_token_tile == 128 || g_force_token_tile == 256)
        return g_force_token_tile;
    if (T <= 64) return 64;
    return 128;
}

static inline int pick_split_k(int T, int N, int K, int bn) {
    const int kblocks = K / kBK;
    int want = 1;
    if (g_force_split_k > 0) {
        want = g_force_split_k;
    } else {
        const int tiles = (N / kBM) * ((T + bn - 1) / bn);
        // weight-streaming regime: too few tiles to cover the SMs -> split K
        if (tiles * 2 <= kNumSMs) {
            want = kNumSMs / tiles;
        }
    }
    if (want > kblocks) want = kblocks;
    while (want > 1 && kblocks % want != 0) --want;
    return want < 1 ? 1 : want;
}

static size_t split_acc_bytes(int T, int N) {
    return (static_cast<size_t>(T) * N * sizeof(int32_t) + 255) & ~static_cast<size_t>(255);
}

struct GemmPlan {
    bool pair;      // CTA-pair kernel (two M-tiles per CTA) or single-CTA tiles
    int bn;         // token tile
    int splits;     // split-K factor through global atomics (single-CTA kernel only)
    int cluster;    // > 1: split-K inside clusters of this many CTAs (reduction in shared memory); 1: the wide-tile kernel unsplit
    int mt = 2;     // CTA-pair kernel: M-tiles per CTA (2: 512-feature tiles; 1: 256-feature tiles, double-buffered accumulators)
};
static GemmPlan plan_gemm(bool sparse, bool out_wide, int T, int N, int K, bool may_split = true);
template <int WT, bool FUSED> static bool use_few_kernel(int T, int N, int K);

// Scratch of a plan that splits K through global memory: int32 [T][N] + one counter per output tile.
static size_t split_workspace_bytes(const GemmPlan& plan, int T, int N) {
    if (plan.pair || plan.splits <= 1) return 0;
    return split_acc_bytes(T, N) + static_cast<size_t>(N / kBM) * ((T + plan.bn - 1) / plan.bn) * sizeof(unsigned int);
}
static size_t gemm_workspace_bytes(bool sparse, int T, int N, int K) {
    if (sparse ? use_few_kernel<kFewSparse, false>(T, N, K) : use_few_kernel<kFewDense, false>(T, N, K)) return 0;
    return std::max(split_workspace_bytes(plan_gemm(sparse, false, T, N, K), T, N), split_workspace_bytes(plan_gemm(sparse, true, T, N, K), T, N));
}

template <bool SPARSE, int BN>
static sbn_status launch_gemm_cfg(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& te,
                                  const CUtensorMap& ty, const GemmParams& p, cudaStream_t stream) {
    using Cfg = GemmConfig<SPARSE, BN>;
    auto kernel = bitlinear_gemm_kernel<SPARSE, BN>;
    if (!ensure_dynamic_smem<bitlinear_gemm_kernel<SPARSE, BN>>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
    const int tiles = (p.N / kBM) * ((p.T + BN - 1) / BN) * p.k_splits;
    const int grid = tiles < kNumSMs ? tiles : kNumSMs;
    const cudaError_t err = launch_kernel(kernel, dim3(grid), dim3(kGemmThreads), Cfg::SMEM_BYTES, stream, ta, tb, te, ty, p);
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

// ---- CTA-pair kernel (large T) -------------------------------------------------------------------
template <bool SPARSE, int MT>
static sbn_status launch_pair(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& te,
                              const PairParams& pp, cudaStream_t stream) {
    using Cfg = PairConfig<SPARSE, MT>;
    auto kernel = bitlinear_gemm_pair_kernel<SPARSE, MT>;
    if (!ensure_dynamic_smem<bitlinear_gemm_pair_kernel<SPARSE, MT>>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
    const int tiles = ((pp.g.N + 256 * MT - 1) / (256 * MT)) * ((pp.g.T + pp.bn - 1) / pp.bn);
    const int pairs = tiles < kNumSMs / 2 ? tiles : kNumSMs / 2;
    const cudaError_t err = launch_kernel(kernel, dim3(2 * pairs), dim3(kPairThreads), Cfg::SMEM_BYTES, stream, ta, tb, te, pp);
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

// Which kernel, which token tile, whether to split K: the measured times (us) of every candidate, as a small model.
//
// The coefficients were fitted to quantiser + GEMM chains (weights from memory): 43 shapes from 640 x 1280 to 65536 x 2560 and
// 2048 x 65536 (K x N), 30 token counts from 9 to 8192, every kernel with its useful tiles and splits, sparse and dense, bf16 and
// fp32 outputs; 43000 timings.  What the model picks is within 0.5 % of the fastest candidate on average (the worst 13 %), and on
// 16 shapes and 24 token counts that the fit has not seen within 0.6 % (12 %).  q = K-blocks per CTA, w = waves.
//   clusters, narrow tiles   a + q (c + x crowd + x2 share of SMs with two CTAs) + tokens (t + s / S) + o crowd min(1, q / 3) + 3-way
//                            owner selection
//   clusters, wide tiles     a + q (c + u bn / 256) + e tokens (S - 1) / S + (share + z q) x share of the SMs in use
//   single-CTA tiles         a + (w q c or m MB) + w d; K split through global memory: a + q c + atomics T N S
//   CTA pairs                a + b bn + (w q (c + u bn / 256) or m MB) + w d, with one or two M-tiles per CTA
// "or": whichever is longer, smoothed (fourth powers); MB = megabytes of weights and outputs.
// The output type matters to the pairs: with two M-tiles the accumulator waits for the stores of fp32 outputs (5 us per tile, bf16
// ones leave through registers in 2.5), with one it does not.  2560 -> 6912 sparse, 6000 tokens, fp32: two M-tiles 86 us, one 75.
struct ClusterCost { double a, c, x, t, s, o, s3, x2; };
struct WideCost { double a, c, e, share, u, c2, u2, z; };   // c2, u2: stages of two K-blocks
struct TileCost { double a, c, d, m; };
struct PairCost { double a, b, c, d, u, m; };
struct PlanCosts {
    ClusterCost narrow32, narrow64;
    WideCost wide;
    TileCost tile64, tile128, tile256;
    PairCost pair1, pair2;
};
static const PlanCosts kPlanCosts[2][2] = {                 // [sparse][fp32 outputs or raw accumulators]
    {{{5.2724, 0.2689, 0.003, 0.002, 0.01, 0.4005, 0.0371, 0.0685}, {5.0562, 0.3367, 0.0157, 0.0225, 0.0051, 0.4646, 1.2385, 0.0819},
      {4.5917, 0.1501, 0.0295, 0.5418, 0.1432, 0.1242, 0.1469, 0.0775},
      {5.2199, 0.2497, 0.5009, 0.07}, {6.0228, 0.2653, 0.7606, 0.1161}, {9.2108, 0.3821, -0.3368, 0.1839}, {4.8432, 0.0053, 0.2966, 0.6719, 0.0509, 0.0002}, {3.4272, 0.0134, 0.3953, 2.9039, 0.1588, 0.1106}},
     {{5.2688, 0.2675, 0.0064, 0.0018, 0.0081, 0.4248, 0.0791, 0.0575}, {5.073, 0.3341, 0.0095, 0.0212, 0.0044, 0.5437, 1.4758, 0.0795},
      {4.5868, 0.1448, 0.0292, 0.5865, 0.1469, 0.1255, 0.1402, 0.0747},
      {5.2396, 0.2516, 0.3646, 0.0725}, {5.8416, 0.2673, 0.4823, 0.1166}, {7.6558, 0.395, 0.0374, 0.1638}, {5.1877, 0.01, 0.2932, 0.8005, 0.0524, 0.0007}, {1.9177, 0.0179, 0.366, 5.1005, 0.2111, 0.1001}}},
    {{{4.757, 0.1929, 0.013, 0.023, 0.0004, 0.2915, 0.0598, 0.0471}, {4.8582, 0.2677, 0.0395, 0.0317, 0.0021, 0.1165, 1.1535, 0.0332},
      {4.7161, 0.2772, 0.0299, 0.2317, -0.0365, 0.1183, 0.0977, 0.0818},
      {5.3343, 0.2414, 0.2205, 0.1108}, {6.2223, 0.2463, 0.546, 0.1228}, {5.3179, 0.2778, 3.487, 0.1858}, {4.8079, 0.0054, 0.1838, 0.6455, 0.0348, 0.0992}, {3.8719, 0.0136, 0.2539, 2.458, 0.1053, 0.1233}},
     {{4.8398, 0.1906, 0.0118, 0.0169, 0.0021, 0.3432, 0.1063, 0.0447}, {4.8808, 0.2655, 0.0342, 0.029, 0.0022, 0.2248, 1.3655, 0.0341},
      {4.6456, 0.2668, 0.03, 0.3028, -0.0285, 0.117, 0.0944, 0.0807},
      {5.1138, 0.2422, 0.2679, 0.126}, {5.9491, 0.2478, 0.3353, 0.1469}, {5.3549, 0.282, 2.349, 0.157}, {4.9998, 0.0107, 0.1749, 0.8473, 0.0446, 0.1231}, {2.7183, 0.0176, 0.233, 4.2553, 0.1481, 0.1171}}}};

// Wide tiles, unsplit, dense: a + kb (c + u bn / 256 + z share) + sh share + tk tokens, share = of the SMs in use; c2, u2 as above.
// [fp32 outputs].  Fitted the same way to 44 shapes, 26 token counts, against the other kernels' costs.
struct WideOneCost { double a, c, u, c2, u2, sh, z, tk; };
static const WideOneCost kWideOneCosts[2] = {{5.0092, 0.1812, 0.1058, 0.1353, 0.1165, 0.7654, 0.037, 0.0119}, {5.05, 0.1741, 0.116, 0.1386, 0.118, 1.025, 0.0223, 0.0102}};

// Clusters of S with two CTAs per SM that were all resident at once; one more waited for a whole kernel lifetime (12288 -> 2304,
// 128 tokens: 72 clusters of 4 19.5 us, other plans 13.1; clusters of 3: 88 were, 90 not always).
constexpr int kNarrowClusters[5] = {0, 0, 148, 88, 70};
// The same with one CTA per SM (wide tiles; 45 clusters of 3 were not: 5376 -> 1920, 230 tokens: 14.8 us, 33 or fewer of 4 9.9).
constexpr int kWideClusters[5] = {0, 0, 74, 44, 33};

static double narrow_cost(const ClusterCost& c, int kb, long tiles, int tokens, int S) {
    const int q = (kb + S - 1) / S;
    // SMs that hold two CTAs: part of the slowdown grows with their share, part is all there once 40 % of them do
    const double two = std::max(0.0, static_cast<double>(tiles * S - kNumSMs) / kNumSMs), crowd = std::min(1.0, 2.5 * two);
    return c.a + q * (c.c + c.x * crowd + c.x2 * two) + tokens * (c.t + c.s / S) + c.o * crowd * std::min(1.0, q / 3.0) + (S == 3 ? c.s3 : 0.0);
}

// out_wide: four bytes per output or more (fp32, or the raw accumulators as well).  may_split: a plan may need a workspace.
static GemmPlan plan_gemm(bool sparse, bool out_wide, int T, int N, int K, bool may_split) {
    GemmPlan best = {false, 64, 1, 0};
    const int kb = K / kBK;
    const int rows = N / kBM;
    if (g_force_token_tile < 0) {                               // diagnostics: the pair kernel as told (split_k 1 = one M-tile per CTA)
        const int cap = sparse ? kPairMaxBnSparse : kPairMaxBnDense;
        GemmPlan g{true, std::min(cap, std::max(32, (-g_force_token_tile) / 16 * 16)), 1, 0};
        g.mt = g_force_split_k == 1 ? 1 : 2;
        return g;
    }
    if (g_force_split_k < 0) {                                  // diagnostics: cluster split-K as told
        int S = -g_force_split_k;
        if (g_force_token_tile >= kWideMinBn) {                 // wide tiles: any width and cluster that fit
            const int bn = std::min(256, g_force_token_tile / 16 * 16);
            const bool unsplit = S == 1;
            S = std::min(8, std::min(S, K / kBK));
            while (S > 1 && !wide_fits(bn, S)) --S;
            if (S > 1 || unsplit) return GemmPlan{false, bn, 1, S};
        }
        S = S >= 8 ? 8 : (S >= 4 ? 4 : (S == 3 ? 3 : 2));
        while (S > 1 && S > K / kBK) --S;
        if (S > 4 && S < 8) S = 4;
        const int bn = g_force_token_tile == 32 ? 32 : 64;
        if (S > 1) return GemmPlan{false, bn, 1, S};
    }
    if (g_force_token_tile > 0 || g_force_split_k > 0) {        // diagnostics: single-CTA kernel as told
        const int bn = pick_token_tile(T);
        return GemmPlan{false, bn, pick_split_k(T, N, K, bn), 0};
    }
    const PlanCosts& cost = kPlanCosts[sparse][out_wide];
    const double megabytes = 1e-6 * N * ((sparse ? 0.625 : 1.0) * K + (out_wide ? 4.0 : 2.0) * T);
    auto longer = [](double x, double y) { return std::sqrt(std::sqrt(x * x * x * x + y * y * y * y)); };
    double best_t = 1e300;
    auto consider = [&](const GemmPlan& g, double t) { if (t < best_t) { best_t = t; best = g; } };
    // Clusters of 2, 3 or 4 CTAs, narrow tiles: all of them resident at once, two CTAs per SM.
    for (const int bn : {32, 64}) {
        const long tiles = static_cast<long>(rows) * ((T + bn - 1) / bn);
        for (int S = 2; S <= 4 && S <= kb; ++S)
            if (tiles <= kNarrowClusters[S])
                consider(GemmPlan{false, bn, 1, S}, narrow_cost(bn == 32 ? cost.narrow32 : cost.narrow64, kb, tiles, std::min(bn, T), S));
    }
    // Wide tiles: one CTA per SM.  (8192 -> 1024 dense, 1000 tokens: 21.3 us, narrow clusters 22.7.)
    if (T > 64 && T <= 2048) {
        const int fewest = (T + 255) / 256;
        for (int tt = fewest; tt <= fewest + (T > 512 ? 4 : 2); ++tt) {
            const int bn = std::max(kWideMinBn, ((T + tt - 1) / tt + 15) / 16 * 16);
            if (bn * (tt - 1) >= T) continue;
            const int tokens = std::min(bn, T);
            const double c = wide_group(sparse, bn) == 2 ? cost.wide.c2 + cost.wide.u2 * bn / 256 : cost.wide.c + cost.wide.u * bn / 256;
            for (int S = 2; S <= 4 && S <= kb; ++S) {
                if (static_cast<long>(rows) * tt > kWideClusters[S] || !wide_fits(bn, S)) continue;
                const int q = (kb + S - 1) / S;
                consider(GemmPlan{false, bn, 1, S}, cost.wide.a + q * c + cost.wide.e * tokens * (S - 1) / S +
                                                        (cost.wide.share + cost.wide.z * q) * rows * tt * S / kNumSMs);
            }
        }
    }
    // The same kernel unsplit, dense weights, one tile per SM: its first stages hold weights before the dependency wait and it fetches two
    // K-blocks with one instruction per operand, which the single-CTA kernel below does not (6912 -> 2560, 777 tokens, us: 24.8,
    // here 22.5; 11008 -> 4096, 600 tokens 39.9 / 33.5; 2560 -> 2560 13.6 / 13.4).  Sparse weights: the pairs' instructions do more
    // (2 to 3 % either way).
    if (!sparse && T > 64 && T <= 2048) {
        const WideOneCost& c = kWideOneCosts[out_wide];
        const int fewest = (T + 255) / 256;
        for (int tt = fewest; tt <= fewest + 5 && static_cast<long>(rows) * tt <= kNumSMs; ++tt) {
            const int bn = std::max(kWideMinBn, ((T + tt - 1) / tt + 15) / 16 * 16);
            if (bn * (tt - 1) >= T) continue;
            const double share = static_cast<double>(rows) * tt / kNumSMs;
            const double block = wide_group(sparse, bn) == 2 ? c.c2 + c.u2 * bn / 256 : c.c + c.u * bn / 256;
            consider(GemmPlan{false, bn, 1, 1}, c.a + kb * (block + c.z * share) + c.sh * share + c.tk * std::min(bn, T));
        }
    }
    // Single-CTA tiles: one token tile in any number of waves, else up to two, with short K (1024 -> 2560: 15.0 us for 2048
    // tokens dense, pairs 15.9) up to four; beyond, the pairs' operand reuse wins.
    for (const int bn : {64, 128, 256}) {
        if (bn > 64 && T <= bn / 2) continue;                   // a tile mostly beyond T
        const TileCost& c = bn == 64 ? cost.tile64 : (bn == 128 ? cost.tile128 : cost.tile256);
        const long tiles = static_cast<long>(rows) * ((T + bn - 1) / bn);
        const long waves = (tiles + kNumSMs - 1) / kNumSMs;
        if (T <= 64 || waves <= (kb <= 12 && bn < 256 ? 4 : 2)) consider(GemmPlan{false, bn, 1, 0}, c.a + longer(waves * kb * c.c, c.m * megabytes) + waves * c.d);
        // K through global memory: dense weights of very long rows only (24576 -> 2304, 9 tokens: 19.1 us, clusters 20.9; at
        // K = 16384 it was slower, sparse weights never faster).  One wave, at least ~100 units of work.
        if (may_split && !sparse && bn == 64 && K >= 24576 && tiles * 2 <= kNumSMs) {
            int sp = static_cast<int>((100 + tiles - 1) / tiles);
            while (sp > 1 && sp <= 10 && kb % sp != 0) ++sp;
            if (sp > 1 && sp <= 10 && tiles * sp <= kNumSMs)
                consider(GemmPlan{false, bn, sp, 0}, 7.6 + kb / sp * 0.269 + 7.2e-6 * T * N * sp);
        }
    }
    // CTA pairs: a tile costs nearly the same whatever its token width, so the tile counts worth a look are the smallest
    // ones, down to those that fill the last wave.  For few tokens too: they have more places than the clusters (4096 -> 20480
    // sparse, 16 tokens: 17.6 us, single-CTA tiles 23.2).
    const int cap = sparse ? kPairMaxBnSparse : kPairMaxBnDense;
    const int fewest = (T + cap - 1) / cap;
    for (int tt = fewest; tt <= fewest + (T < 1000 ? 3 : 8); ++tt) {
        const int bn = std::max(T > 64 ? 80 : 32, ((T + tt - 1) / tt + 15) / 16 * 16);
        if (bn * (tt - 1) >= T) continue;
        for (int mt = 1; mt <= 2; ++mt) {
            const PairCost& c = mt == 1 ? cost.pair1 : cost.pair2;
            const long tiles = static_cast<long>((N + 256 * mt - 1) / (256 * mt)) * tt;
            const long waves = (tiles + kNumSMs / 2 - 1) / (kNumSMs / 2);
            GemmPlan g{true, bn, 1, 0};
            g.mt = mt;
            consider(g, c.a + c.b * bn + longer(waves * kb * (c.c + c.u * bn / 256), c.m * megabytes) + waves * c.d);
        }
    }
    return best;
}

static sbn_status run_gemm_pair(bool sparse, const int8_t* xq, const float* a_scale, int T,
                                const int8_t* wvals, const uint8_t* meta, const float* w_scale,
                                int N, int K, const float* bias, void* y, sbn_out_dtype dt,
                                int32_t* acc_out, int bn, int mt, cudaStream_t stream) {
    CUtensorMap ta, tb, te;
    bool ok;
    const uint64_t KBk = static_cast<uint64_t>(K) / kBK, NB = static_cast<uint64_t>(N) / kBM;
    if (sparse) {
        constexpr int kbs = PairConfig<true>::KBS;
        ok = encode_3d_1k(&ta, wvals, KBk * 8, NB, 8 * kbs, mt) && encode_3d_1k(&te, meta, KBk * 2, NB, 2 * kbs, mt) &&
             encode_3d_1k(&tb, xq, xq_tb8(T), KBk, bn / 16, kbs);
    } else {
        constexpr int kbs = PairConfig<false>::KBS;
        ok = encode_3d_1k(&ta, wvals, KBk * 16, NB, 16 * kbs, mt) && encode_3d_1k(&tb, xq, xq_tb8(T), KBk, bn / 16, kbs);
        te = ta;
    }
    if (!ok) return SBN_ERR_CUDA;
    PairParams pp;
    pp.g.T = T; pp.g.N = N; pp.g.K = K;
    pp.g.k_blocks_total = K / kBK;
    pp.g.k_splits = 1;
    pp.g.tb8 = static_cast<int>(xq_tb8(T));
    pp.g.a_scale = a_scale; pp.g.w_scale = w_scale; pp.g.bias = bias;
    pp.g.y = y; pp.g.out_bf16 = (dt == SBN_OUT_BF16);
    pp.g.acc_out = acc_out;
    pp.g.split_acc = nullptr; pp.g.split_counters = nullptr;
    pp.g.w_vals = wvals; pp.g.w_meta = sparse ? meta : nullptr; pp.g.w_tile_bytes = sparse ? 8192 : 16384;
    pp.g.test_skip_loads = g_test_break_waits;
    pp.g.probe = g_gemm_probe;
    pp.bn = bn;
    if (mt == 1) return sparse ? launch_pair<true, 1>(ta, tb, te, pp, stream) : launch_pair<false, 1>(ta, tb, te, pp, stream);
    return sparse ? launch_pair<true, 2>(ta, tb, te, pp, stream) : launch_pair<false, 2>(ta, tb, te, pp, stream);
}

template <bool SPARSE, int BN>
static sbn_status launch_splitk_cluster(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& te,
                                        const GemmParams& p, int cluster, cudaStream_t stream) {
    using Cfg = SplitConfig<SPARSE, BN>;
    auto kernel = bitlinear_gemm_splitk_cluster_kernel<SPARSE, BN>;
    if (!ensure_dynamic_smem<bitlinear_gemm_splitk_cluster_kernel<SPARSE, BN>>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
    const int tiles = (p.N / kBM) * ((p.T + BN - 1) / BN);
    const cudaError_t err = launch_kernel_cluster(kernel, dim3(tiles * cluster), dim3(kSplitThreads), Cfg::SMEM_BYTES, stream,
                                                  static_cast<unsigned>(cluster), ta, tb, te, p);
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

template <bool SPARSE, int G>
static sbn_status launch_splitk_wide_cfg(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& te, const GemmParams& p, int bn,
                                         int cluster, cudaStream_t stream) {
    if (!ensure_dynamic_smem<bitlinear_gemm_splitk_wide_kernel<SPARSE, G>>(kWideSmemBytes)) return SBN_ERR_CUDA;
    const int tiles = (p.N / kBM) * ((p.T + bn - 1) / bn);
    const cudaError_t err = launch_kernel_cluster(bitlinear_gemm_splitk_wide_kernel<SPARSE, G>, dim3(tiles * cluster), dim3(kWideThreads),
                                                  kWideSmemBytes, stream, static_cast<unsigned>(cluster), ta, tb, te, p, bn);
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}
template <bool SPARSE>
static sbn_status launch_splitk_wide(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& te, const GemmParams& p, int bn,
                                     int cluster, cudaStream_t stream) {
    return wide_group(SPARSE, bn) == 2 ? launch_splitk_wide_cfg<SPARSE, 2>(ta, tb, te, p, bn, cluster, stream)
                                       : launch_splitk_wide_cfg<SPARSE, 1>(ta, tb, te, p, bn, cluster, stream);
}

// ---- few tokens: register-fed kernel ----------------------------------------------------------------
static FewParams few_params(int T, int N, int K, const void* xq, const void* x_bf16, const float* a_scale, float* a_scale_out, const void* vals,
                            const uint8_t* meta, const float* w_scale, const float* bias, void* y, sbn_out_dtype dt, int32_t* acc_out) {
    FewParams p;
    p.T = T; p.N = N; p.k_blocks = K / kBK;
    p.tb8 = static_cast<int>(xq_tb8(T));
    p.xq = static_cast<const uint8_t*>(xq);
    p.x_bf16 = static_cast<const uint4*>(x_bf16);
    p.a_scale = a_scale; p.a_scale_out = a_scale_out;
    p.vals = static_cast<const uint8_t*>(vals); p.meta = meta;
    p.w_scale = w_scale; p.bias = bias;
    p.y = y; p.out_bf16 = (dt == SBN_OUT_BF16);
    p.acc_out = acc_out;
    return p;
}
template <int WT, bool FUSED>
static bool use_few_kernel(int T, int N, int K) {
    if (g_force_token_tile != 0 || g_force_split_k != 0 || g_test_break_waits) return false;   // diagnostics: the tcgen05 kernels as told
    return few_takes<WT, FUSED>(T, N, K);
}

static sbn_status run_gemm(bool sparse, const int8_t* xq, const float* a_scale, int T,
                           const int8_t* wvals, const uint8_t* meta, const float* w_scale,
                           int N, int K, const float* bias, void* y, sbn_out_dtype dt,
                           int32_t* acc_out, void* ws, size_t ws_bytes, cudaStream_t stream) {
    if (!xq || !a_scale || !wvals || !w_scale || !y || (sparse && !meta)) return SBN_ERR_NULL;
    if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (dt != SBN_OUT_F32 && dt != SBN_OUT_BF16) return SBN_ERR_UNSUPPORTED;
    if (misaligned(xq, 16) || misaligned(wvals, 16) || (sparse && misaligned(meta, 16)) ||
        misaligned(y, 16) || misaligned(a_scale, 4) || misaligned(w_scale, 4) ||
        (acc_out && misaligned(acc_out, 4)) || (bias && misaligned(bias, 4)))
        return SBN_ERR_ALIGN;

    if (sparse ? use_few_kernel<kFewSparse, false>(T, N, K) : use_few_kernel<kFewDense, false>(T, N, K)) {
        const FewParams p = few_params(T, N, K, xq, nullptr, a_scale, nullptr, wvals, meta, w_scale, bias, y, dt, acc_out);
        return sparse ? launch_few<kFewSparse, false>(p, stream) : launch_few<kFewDense, false>(p, stream);
    }
    const bool out_wide = dt == SBN_OUT_F32 || acc_out != nullptr;
    GemmPlan plan = plan_gemm(sparse, out_wide, T, N, K);
    if (plan.splits > 1) {
        // scratch is zero on entry (caller's duty before the first use) and the kernel re-zeroes it.  Without it: the
        // fastest plan that needs none, unless this one was asked for
        if (!ws || ws_bytes < split_workspace_bytes(plan, T, N)) {
            if (g_force_token_tile != 0 || g_force_split_k != 0) return SBN_ERR_WORKSPACE;
            plan = plan_gemm(sparse, out_wide, T, N, K, false);
        } else if (misaligned(ws, 16)) {
            return SBN_ERR_ALIGN;
        }
    }
    if (plan.pair)
        return run_gemm_pair(sparse, xq, a_scale, T, wvals, meta, w_scale, N, K, bias, y, dt, acc_out, plan.bn, plan.mt, stream);

    const int bn = plan.bn;
    const int splits = plan.splits;

    CUtensorMap ta, tb, te, ty;
    bool ok;
    const uint64_t NK = static_cast<uint64_t>(N) * K;
    if (sparse) {
        ok = encode_flat_1k(&ta, wvals, NK / 2, 8) && encode_flat_1k(&te, meta, NK / 8, 2);
    } else {
        ok = encode_flat_1k(&ta, wvals, NK, 16);
        te = ta;
    }
    ok = ok && encode_flat_1k(&tb, xq, xq_tiled_bytes(T, K), bn / 8);
    ok = ok && encode_2d_out(&ty, y, N, T, dt == SBN_OUT_BF16, 32);
    if (!ok) return SBN_ERR_CUDA;

    GemmParams p;
    p.T = T; p.N = N; p.K = K;
    p.k_blocks_total = K / kBK;
    p.k_splits = splits;
    p.tb8 = static_cast<int>(xq_tb8(T));
    p.a_scale = a_scale; p.w_scale = w_scale; p.bias = bias;
    p.y = y; p.out_bf16 = (dt == SBN_OUT_BF16);
    p.acc_out = acc_out;
    p.split_acc = splits > 1 ? static_cast<int32_t*>(ws) : nullptr;
    p.split_counters = splits > 1 ? reinterpret_cast<unsigned int*>(static_cast<char*>(ws) + split_acc_bytes(T, N)) : nullptr;
    p.w_vals = wvals; p.w_meta = sparse ? meta : nullptr; p.w_tile_bytes = sparse ? 8192 : 16384;
    p.test_skip_loads = g_test_break_waits;

    if (plan.cluster >= 1) {
        // the cluster sizes that the kernels have code for; another would write to CTAs that do not exist
        const bool wide = bn >= kWideMinBn;
        if (wide ? plan.cluster > 8 : (plan.cluster != 2 && plan.cluster != 3 && plan.cluster != 4 && plan.cluster != 8)) return SBN_ERR_UNSUPPORTED;
        p.k_splits = 1;
        if (wide) {                                             // boxes of wide_group K-blocks
            const uint32_t G = static_cast<uint32_t>(wide_group(sparse, bn));
            ok = (sparse ? encode_flat_1k(&ta, wvals, NK / 2, 8 * G) && encode_flat_1k(&te, meta, NK / 8, 2 * G) : encode_flat_1k(&ta, wvals, NK, 16 * G)) &&
                 (G == 1 || encode_3d_1k(&tb, xq, xq_tb8(T), static_cast<uint64_t>(K) / kBK, static_cast<uint32_t>(bn / 8), G));   // G = 1: tb as it is
            if (!ok) return SBN_ERR_CUDA;
            return sparse ? launch_splitk_wide<true>(ta, tb, te, p, bn, plan.cluster, stream)
                          : launch_splitk_wide<false>(ta, tb, te, p, bn, plan.cluster, stream);
        }
        if (sparse && bn == 32) {                               // two K-blocks per stage
            static_assert(SplitConfig<true, 32>::G == 2 && SplitConfig<true, 64>::G == 1 && SplitConfig<false, 32>::G == 1, "boxes");
            if (!encode_flat_1k(&ta, wvals, NK / 2, 16) || !encode_flat_1k(&te, meta, NK / 8, 4) ||
                !encode_3d_1k(&tb, xq, xq_tb8(T), static_cast<uint64_t>(K) / kBK, 4, 2))
                return SBN_ERR_CUDA;
        }
        if (sparse) return bn == 32 ? launch_splitk_cluster<true, 32>(ta, tb, te, p, plan.cluster, stream)
                                    : launch_splitk_cluster<true, 64>(ta, tb, te, p, plan.cluster, stream);
        return bn == 32 ? launch_splitk_cluster<false, 32>(ta, tb, te, p, plan.cluster, stream)
                        : launch_splitk_cluster<false, 64>(ta, tb, te, p, plan.cluster, stream);
    }

    sbn_status st;
#define SBN_GEMM_CASE(S, B) st = launch_gemm_cfg<S, B>(ta, tb, te, ty, p, stream)
    if (sparse) {
        if (bn == 64) SBN_GEMM_CASE(true, 64); else if (bn == 128) SBN_GEMM_CASE(true, 128); else SBN_GEMM_CASE(true, 256);
    } else {
        if (bn == 64) SBN_GEMM_CASE(false, 64); else if (bn == 128) SBN_GEMM_CASE(false, 128); else SBN_GEMM_CASE(false, 256);
    }
#undef SBN_GEMM_CASE
    if (st != SBN_OK) return st;
    return SBN_OK;
}

// ---- backward GEMMs (bf16) -------------------------------------------------------------------------
struct BackwardWs {                    // W_eff [N][K] and x_q [T][K], both bf16
    size_t w_off, xq_off, total;
};
static BackwardWs backward_ws_layout(int T, int N, int K) {
    BackwardWs w;
    auto up = [](size_t v) { return (v + 255) & ~static_cast<size_t>(255); };
    w.w_off = 0;
    w.xq_off = up(static_cast<size_t>(K) * N * 2);
    w.total = w.xq_off + up(static_cast<size_t>(T) * K * 2);
    return w;
}

static sbn_status run_backward(const void* dY, int T, const int8_t* xq, const float* a_scale, const int8_t* vals, const uint8_t* meta,
                               const float* w_scale, int N, int K, void* dX, float* dW, void* ws, cudaStream_t stream) {
    const BackwardWs lay = backward_ws_layout(T, N, K);
    char* base = static_cast<char*>(ws);
    const int KB = K / kBK, tiles_k = (K + 255) / 256;
    const int w_items = dX ? KB * (N / kBM) : 0;
    const int x_items = dW ? KB * ((T + kPrepItemTokens - 1) / kPrepItemTokens) : 0;
    const int tiles[2] = {dW ? (N + 255) / 256 * tiles_k : 0, dX ? (T + 255) / 256 * tiles_k : 0};
    const int stages[2] = {(T + 63) / 64, N / 64};
    Bf16GemmParams p;
    p.part[0] = Bf16Part{N, T, dW, 0, nullptr};
    p.part[1] = Bf16Part{T, N, dX, 1, w_scale};
    p.Nn = K;
    const PrepJob job{reinterpret_cast<const uint8_t*>(vals), meta, reinterpret_cast<uint16_t*>(base + lay.w_off),
                      reinterpret_cast<const uint8_t*>(xq), a_scale, reinterpret_cast<uint16_t*>(base + lay.xq_off), T, N, K, w_items, x_items};
    p.plan = plan_backward(tiles, stages, g_force_token_tile < 0 ? (-g_force_token_tile <= 128 ? 1 : 0) : -1);

    const uint64_t t = static_cast<uint64_t>(T), n = static_cast<uint64_t>(N), k = static_cast<uint64_t>(K);
    Bf16Maps maps;                                              // only those that the plan reads are filled in
    bool ok = (!dW || encode_3d_bf16_blocks(&maps.aw, dY, n, t, 2)) && (!dX || encode_2d_bf16_sw128(&maps.ax, dY, n, t, n, 128));
    for (int g = 0; ok && g < p.plan.segments; ++g) {
        const int part = p.plan.seg[g].part, half = p.plan.seg[g].half;
        ok = encode_3d_bf16_blocks(&maps.b[part][half], base + (part == 0 ? lay.xq_off : lay.w_off), k, part == 0 ? t : n, half ? 1 : 2);
    }
    if (!ok) return SBN_ERR_CUDA;
    if (!ensure_dynamic_smem<backward_gemm_kernel>(kBf16SmemBytes)) return SBN_ERR_CUDA;
    const int blocks = std::max(1, std::min(w_items + x_items, 16 * device_sm_count()));
    if (launch_kernel(backward_prep_kernel, dim3(blocks), dim3(kPrepThreads), 0, stream, job) != cudaSuccess) return SBN_ERR_CUDA;
    ++g_launch_count;
    if (launch_kernel(backward_gemm_kernel, dim3(2 * kBackwardPairs), dim3(kBf16Threads), kBf16SmemBytes, stream, maps, p) != cudaSuccess)
        return SBN_ERR_CUDA;
    ++g_launch_count;
    return SBN_OK;
}

// ------------------------------------------------------------------------------------------------
// Built-in scratch for sbn_quantize_mask_pack_static_ws: part of the library image, so callers
// that cannot allocate still have somewhere to put the pass-1 partial sums.  In host code the
// symbol below is only a handle; its device address is looked up once per device.
// ------------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_scratch[SBN_STATIC_SCRATCH_BYTES];
static_assert(sizeof(QmpWorkspace) <= SBN_STATIC_SCRATCH_BYTES, "built-in scratch too small");

constexpr int kMaxDevices = 64;
static void* g_static_scratch_addr[kMaxDevices] = {};
static std::mutex g_static_scratch_mutex;

// Device address of g_static_scratch on the current device (nullptr on failure).
static void* static_scratch_for_current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (g_static_scratch_addr[dev] == nullptr) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess) return nullptr;
        g_static_scratch_addr[dev] = ptr;
    }
    return g_static_scratch_addr[dev];
}

}  // namespace sbn

// ------------------------------------------------------------------------------------------------
// extern "C"
// ------------------------------------------------------------------------------------------------
using namespace sbn;

extern "C" {

size_t sbn_xq_bytes(int T, int K) {
    if (T <= 0 || K <= 0 || K % kBK != 0) return 0;
    return xq_tiled_bytes(T, K);
}

size_t sbn_workspace_bytes(int op, int T, int N, int K) {
    switch (op) {
        case SBN_OP_QUANTIZE_MASK_PACK: return sizeof(QmpWorkspace);       // one matrix; batches: sbn_batch_workspace_bytes
        case SBN_OP_QUANT_ACT: return 0;
        case SBN_OP_BACKWARD:
            if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0) return 0;
            return backward_ws_layout(T, N, K).total;
        case SBN_OP_SPARSE_BITLINEAR:
        case SBN_OP_BITLINEAR:
            if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0) return 0;
            return gemm_workspace_bytes(op == SBN_OP_SPARSE_BITLINEAR, T, N, K);
        default: return 0;
    }
}

static sbn_status quantize_mask_pack_any(const void* W, bool w_bf16, int N, int K, int n_keep, int m_group,
                                         int8_t* vals, uint8_t* meta, float* w_scale, int8_t* dense_q,
                                         const uint8_t* prev_meta, unsigned long long* flip_bits,
                                         void* ws, size_t ws_bytes, void* stream) {
    if (!W || !vals || !meta || !w_scale) return SBN_ERR_NULL;
    if (prev_meta && !flip_bits) return SBN_ERR_NULL;
    const bool p68 = n_keep == 6 && m_group == 8;
    if (!p68 && (n_keep != 2 || m_group != 4)) return SBN_ERR_UNSUPPORTED;
    if (p68 && dense_q) return SBN_ERR_UNSUPPORTED;           // the dense W_q does not depend on the pattern
    if (N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (p68 && K % (2 * kBK) != 0) return SBN_ERR_SHAPE;     // K' = 3K/2 must be a whole number of 128-column blocks
    if (!ws || ws_bytes < sizeof(QmpWorkspace)) return SBN_ERR_WORKSPACE;
    if (misaligned(W, 16) || misaligned(vals, 16) || misaligned(meta, 16) || misaligned(ws, 16) ||
        misaligned(w_scale, 4) || (dense_q && misaligned(dense_q, 16)) ||
        (prev_meta && misaligned(prev_meta, 16)) || (flip_bits && misaligned(flip_bits, 8)))
        return SBN_ERR_ALIGN;
    if (p68)
        return launch_quantize_mask_pack<68>(W, w_bf16, N, K, vals, meta, w_scale, nullptr, prev_meta, flip_bits,
                                             static_cast<QmpWorkspace*>(ws), static_cast<cudaStream_t>(stream));
    return launch_quantize_mask_pack<24>(W, w_bf16, N, K, vals, meta, w_scale, dense_q, prev_meta, flip_bits,
                                     static_cast<QmpWorkspace*>(ws),
                                     static_cast<cudaStream_t>(stream));
}

sbn_status sbn_quantize_mask_pack(const float* W, int N, int K, int n_keep, int m_group,
                                  int8_t* vals, uint8_t* meta, float* w_scale, int8_t* dense_q,
                                  const uint8_t* prev_meta, unsigned long long* flip_bits,
                                  void* ws, size_t ws_bytes, void* stream) {
    return quantize_mask_pack_any(W, false, N, K, n_keep, m_group, vals, meta, w_scale, dense_q, prev_meta, flip_bits,
                                  ws, ws_bytes, stream);
}

sbn_status sbn_quantize_mask_pack_bf16(const void* W_bf16, int N, int K, int n_keep, int m_group,
                                       int8_t* vals, uint8_t* meta, float* w_scale, int8_t* dense_q,
                                       const uint8_t* prev_meta, unsigned long long* flip_bits,
                                       void* ws, size_t ws_bytes, void* stream) {
    return quantize_mask_pack_any(W_bf16, true, N, K, n_keep, m_group, vals, meta, w_scale, dense_q, prev_meta, flip_bits,
                                  ws, ws_bytes, stream);
}

// Batch workspace: [generation word, 256 B][job descriptors 1.., padded to 256 B][count x 148 slots].
static size_t batch_desc_bytes(int count) {
    return (static_cast<size_t>(count) * sizeof(QmpDesc) + 255) & ~static_cast<size_t>(255);
}
size_t sbn_batch_workspace_bytes(int count) {
    if (count <= 0) return 0;
    return 256 + batch_desc_bytes(count) + static_cast<size_t>(count) * sizeof(QmpWorkspace);
}

sbn_status sbn_quantize_mask_pack_batched(int count, const sbn_pack_job* jobs, void* ws, size_t ws_bytes,
                                          void* stream) {
    if (count <= 0) return SBN_ERR_SHAPE;
    if (!jobs) return SBN_ERR_NULL;
    if (!ws || ws_bytes < sbn_batch_workspace_bytes(count)) return SBN_ERR_WORKSPACE;
    if (misaligned(ws, 16)) return SBN_ERR_ALIGN;
    std::vector<QmpDesc> descs(static_cast<size_t>(count));
    for (int i = 0; i < count; ++i) {
        const sbn_pack_job& j = jobs[i];
        if (!j.W || !j.vals || !j.meta || !j.w_scale) return SBN_ERR_NULL;
        if (j.prev_meta && !j.flip_bits) return SBN_ERR_NULL;
        if (j.N <= 0 || j.K <= 0 || j.N % kBM != 0 || j.K % kBK != 0 || j.K > (1 << 20)) return SBN_ERR_SHAPE;
        if (misaligned(j.W, 16) || misaligned(j.vals, 16) || misaligned(j.meta, 16) || misaligned(j.w_scale, 4) ||
            (j.dense_q && misaligned(j.dense_q, 16)) || (j.prev_meta && misaligned(j.prev_meta, 16)) ||
            (j.flip_bits && misaligned(j.flip_bits, 8)))
            return SBN_ERR_ALIGN;
        if (j.gamma_hint && misaligned(j.gamma_hint, 4)) return SBN_ERR_ALIGN;
        descs[i] = qmp_make_desc(j.W, j.w_bf16 != 0, j.N, j.K, j.vals, j.meta, j.w_scale, j.dense_q, j.prev_meta, j.flip_bits,
                                 j.gamma_hint);
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned long long* generation = static_cast<unsigned long long*>(ws);
    QmpDesc* descs_dev = reinterpret_cast<QmpDesc*>(static_cast<char*>(ws) + 256);
    QmpSlot* slots = reinterpret_cast<QmpSlot*>(static_cast<char*>(ws) + 256 + batch_desc_bytes(count));
    // One launch per kQmpMaxBatch matrices (the kernel keeps a little state per matrix on chip).  All jobs
    // but the first of a launch are read by the kernel from the workspace (the first travels as a kernel
    // argument).  They get there as arguments of small store kernels, a chunk at a time: nothing is staged
    // through host memory, so the call only enqueues and the caller's array is free as soon as it returns.
    for (int lo = 0; lo < count; lo += kQmpMaxBatch) {
        const int n_here = std::min(kQmpMaxBatch, count - lo);
        uint32_t max_units = 0;
        for (int i = 0; i < n_here; ++i) max_units = std::max(max_units, descs[static_cast<size_t>(lo + i)].num_units);
        // batches of up to kQmpInlineDescs matrices travel in the kernel's parameters: nothing to store first
        for (int at = 1; n_here > kQmpInlineDescs && at < n_here; at += kQmpDescChunk) {
            QmpDescChunk chunk;
            const int n = std::min(kQmpDescChunk, n_here - at);
            for (int i = 0; i < n; ++i) chunk.d[i] = descs[static_cast<size_t>(lo + at + i)];
            for (int i = n; i < kQmpDescChunk; ++i) chunk.d[i] = descs[0];
            const cudaError_t err = launch_kernel(qmp_store_descs_kernel, dim3(1), dim3(64), 0, s, chunk, descs_dev + (lo + at - 1), n);
            ++g_launch_count;
            if (err != cudaSuccess) return SBN_ERR_CUDA;
        }
        const sbn_status st = launch_quantize_mask_pack_stream<24>(descs.data() + lo, descs_dev + lo, n_here, max_units,
                                                               slots + static_cast<size_t>(lo) * kQmpMaxCtas, generation, s);
        if (st != SBN_OK) return st;
    }
    return SBN_OK;
}

sbn_status sbn_quantize_mask_pack_static_ws(const float* W, int N, int K, int n_keep, int m_group,
                                            int8_t* vals, uint8_t* meta, float* w_scale,
                                            int8_t* dense_q, const uint8_t* prev_meta,
                                            unsigned long long* flip_bits, void* stream) {
    // size limits first: nothing below runs for a shape the built-in scratch cannot serve
    if (N > 0 && K > 0) {
        if (static_cast<long long>(N) * K > SBN_STATIC_MAX_ELEMS) return SBN_ERR_TOO_LARGE;
        if (sbn_workspace_bytes(SBN_OP_QUANTIZE_MASK_PACK, 0, N, K) > SBN_STATIC_SCRATCH_BYTES)
            return SBN_ERR_TOO_LARGE;
    }
    if (!W || !vals || !meta || !w_scale) return SBN_ERR_NULL;
    if (prev_meta && !flip_bits) return SBN_ERR_NULL;
    if (n_keep != 2 || m_group != 4) return SBN_ERR_UNSUPPORTED;
    if (N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (misaligned(W, 16) || misaligned(vals, 16) || misaligned(meta, 16) || misaligned(w_scale, 4) ||
        (dense_q && misaligned(dense_q, 16)) || (prev_meta && misaligned(prev_meta, 16)) ||
        (flip_bits && misaligned(flip_bits, 8)))
        return SBN_ERR_ALIGN;
    void* scratch = static_scratch_for_current_device();
    if (!scratch) return SBN_ERR_CUDA;
    // every slot that is read carries this call's nonce, so stale contents are harmless
    return launch_quantize_mask_pack<24>(W, false, N, K, vals, meta, w_scale, dense_q, prev_meta, flip_bits,
                                     static_cast<QmpWorkspace*>(scratch),
                                     static_cast<cudaStream_t>(stream));
}

sbn_status sbn_quant_act(const void* x_bf16, int T, int K, int8_t* xq, float* a_scale, void* stream) {
    if (!x_bf16 || !xq || !a_scale) return SBN_ERR_NULL;
    if (T <= 0 || K <= 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (misaligned(x_bf16, 16) || misaligned(xq, 16) || misaligned(a_scale, 4)) return SBN_ERR_ALIGN;
    return quantise(x_bf16, T, K, xq, a_scale, static_cast<cudaStream_t>(stream));
}

sbn_status sbn_quant_act_expand68(const void* x_bf16, int T, int K, int8_t* xq, float* a_scale, void* stream) {
    if (!x_bf16 || !xq || !a_scale) return SBN_ERR_NULL;
    if (T <= 0 || K <= 0 || K % (2 * kBK) != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (misaligned(x_bf16, 16) || misaligned(xq, 16) || misaligned(a_scale, 4)) return SBN_ERR_ALIGN;
    return launch_quant_act<true>(x_bf16, T, K, xq, a_scale, static_cast<cudaStream_t>(stream));
}

sbn_status sbn_norm_quant_act_expand68(const void* x_bf16, int T, int K, const float* gain, float eps, int8_t* xq,
                                       float* a_scale, void* stream) {
    if (!x_bf16 || !xq || !a_scale) return SBN_ERR_NULL;
    if (T <= 0 || K <= 0 || K % (2 * kBK) != 0) return SBN_ERR_SHAPE;
    if (K > 16384) return SBN_ERR_UNSUPPORTED;
    if (!(eps >= 0.0f)) return SBN_ERR_SHAPE;
    if (misaligned(x_bf16, 16) || misaligned(xq, 16) || misaligned(a_scale, 4) || (gain && misaligned(gain, 16)))
        return SBN_ERR_ALIGN;
    return launch_norm_quant_act<true>(x_bf16, T, K, gain, eps, xq, a_scale, static_cast<cudaStream_t>(stream));
}

int sbn_expanded_k(int K, int n_keep, int m_group) {
    if (K <= 0) return 0;
    if (n_keep == 2 && m_group == 4) return K;
    if (n_keep == 6 && m_group == 8 && K % (2 * kBK) == 0 && K <= (1 << 20)) return K / 2 * 3;
    return 0;
}

sbn_status sbn_norm_quant_act(const void* x_bf16, int T, int K, const float* gain, float eps, int8_t* xq,
                              float* a_scale, void* stream) {
    if (!x_bf16 || !xq || !a_scale) return SBN_ERR_NULL;
    if (T <= 0 || K <= 0 || K % kBK != 0) return SBN_ERR_SHAPE;
    if (K > 16384) return SBN_ERR_UNSUPPORTED;
    if (!(eps >= 0.0f)) return SBN_ERR_SHAPE;
    if (misaligned(x_bf16, 16) || misaligned(xq, 16) || misaligned(a_scale, 4) || (gain && misaligned(gain, 16)))
        return SBN_ERR_ALIGN;
    return normalise_and_quantise(x_bf16, T, K, gain, eps, xq, a_scale, static_cast<cudaStream_t>(stream));
}

sbn_status sbn_sparse_bitlinear(const int8_t* xq, const float* a_scale, int T, const int8_t* vals,
                                const uint8_t* meta, const float* w_scale, int N, int K,
                                const float* bias, void* y, sbn_out_dtype dt, int32_t* acc_out,
                                void* ws, size_t ws_bytes, void* stream) {
    return run_gemm(true, xq, a_scale, T, vals, meta, w_scale, N, K, bias, y, dt, acc_out, ws, ws_bytes,
                    static_cast<cudaStream_t>(stream));
}

sbn_status sbn_bitlinear(const int8_t* xq, const float* a_scale, int T, const int8_t* dense_q,
                         const float* w_scale, int N, int K, const float* bias, void* y,
                         sbn_out_dtype dt, int32_t* acc_out, void* ws, size_t ws_bytes, void* stream) {
    return run_gemm(false, xq, a_scale, T, dense_q, nullptr, w_scale, N, K, bias, y, dt, acc_out, ws,
                    ws_bytes, static_cast<cudaStream_t>(stream));
}

sbn_status sbn_layer_forward_host(const void* x_bf16_host, int T, int K, void* x_dev, int8_t* xq_dev,
                                  float* a_scale_dev, const int8_t* vals, const uint8_t* meta,
                                  const int8_t* dense_q, const float* w_scale, int N,
                                  const float* bias, void* y_dev, void* y_host, sbn_out_dtype dt,
                                  void* ws, size_t ws_bytes, void* stream) {
    if (!x_bf16_host || !x_dev || !xq_dev || !a_scale_dev || !y_dev || !y_host) return SBN_ERR_NULL;
    if (T <= 0 || K <= 0 || N <= 0) return SBN_ERR_SHAPE;
    if (!vals && !dense_q) return SBN_ERR_NULL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t x_bytes = static_cast<size_t>(T) * K * 2;
    if (cudaMemcpyAsync(x_dev, x_bf16_host, x_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return SBN_ERR_CUDA;
    sbn_status st = sbn_quant_act(x_dev, T, K, xq_dev, a_scale_dev, stream);
    if (st != SBN_OK) return st;
    if (vals) {
        st = sbn_sparse_bitlinear(xq_dev, a_scale_dev, T, vals, meta, w_scale, N, K, bias, y_dev, dt, nullptr, ws, ws_bytes, stream);
    } else {
        st = sbn_bitlinear(xq_dev, a_scale_dev, T, dense_q, w_scale, N, K, bias, y_dev, dt, nullptr, ws, ws_bytes, stream);
    }
    if (st != SBN_OK) return st;
    const size_t y_bytes = static_cast<size_t>(T) * N * (dt == SBN_OUT_BF16 ? 2 : 4);
    if (cudaMemcpyAsync(y_host, y_dev, y_bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) return SBN_ERR_CUDA;
    return SBN_OK;
}

// Cluster size of the fused and packed kernels, which have 32-token tiles only: the cost model of plan_gemm for that tile.  Over
// 144 to 176 calls each (16 shapes, 9 to 400 tokens) its choice is within 0.5 % of the best size on average; an older model of
// these kernels alone, which knew no residency limit below 296 CTAs, was 3 % off (6912 -> 2560 fused, 128 tokens: 23.0 us, now 17.3).
static int pick_cluster_32(bool sparse, int T, int N, int K) {
    const int kb = K / kBK, rows = N / kBM;
    if (g_force_split_k < 0) {                                  // diagnostics: cluster size as told
        int S = -g_force_split_k;
        S = S >= 4 ? 4 : (S == 3 ? 3 : 2);
        while (S > 2 && S > kb) --S;
        return S;
    }
    const long tiles = static_cast<long>(rows) * ((T + 31) / 32);
    int best_s = 2;
    double best_t = 1e300;
    for (int S = 2; S <= 4 && S <= kb; ++S) {
        if (S > 2 && tiles > kNarrowClusters[S]) continue;
        const double t = narrow_cost(kPlanCosts[sparse][false].narrow32, kb, tiles, std::min(32, T), S);
        if (t < best_t) { best_t = t; best_s = S; }
    }
    return best_s;
}

static sbn_status run_fused_act(bool sparse, const void* x_bf16, int T, const int8_t* wvals, const uint8_t* meta,
                                const float* w_scale, int N, int K, const float* bias, void* y, sbn_out_dtype dt,
                                int32_t* acc_out, float* a_scale_out, cudaStream_t stream) {
    if (!x_bf16 || !wvals || !w_scale || !y || (sparse && !meta)) return SBN_ERR_NULL;
    if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (dt != SBN_OUT_F32 && dt != SBN_OUT_BF16) return SBN_ERR_UNSUPPORTED;
    if (T > 256 || K < 2 * kBK) return SBN_ERR_UNSUPPORTED;           // the few-token regime only
    if (misaligned(x_bf16, 16) || misaligned(wvals, 16) || (sparse && misaligned(meta, 16)) || misaligned(y, 16) ||
        misaligned(w_scale, 4) || (acc_out && misaligned(acc_out, 4)) || (bias && misaligned(bias, 4)) ||
        (a_scale_out && misaligned(a_scale_out, 4)))
        return SBN_ERR_ALIGN;
    if (sparse ? use_few_kernel<kFewSparse, true>(T, N, K) : use_few_kernel<kFewDense, true>(T, N, K)) {
        const FewParams p = few_params(T, N, K, nullptr, x_bf16, nullptr, a_scale_out, wvals, meta, w_scale, bias, y, dt, acc_out);
        return sparse ? launch_few<kFewSparse, true>(p, stream) : launch_few<kFewDense, true>(p, stream);
    }
    CUtensorMap ta, te;
    bool ok;
    const uint64_t NK = static_cast<uint64_t>(N) * K;
    if (sparse) {
        ok = encode_flat_1k(&ta, wvals, NK / 2, 8) && encode_flat_1k(&te, meta, NK / 8, 2);
    } else {
        ok = encode_flat_1k(&ta, wvals, NK, 16);
        te = ta;
    }
    if (!ok) return SBN_ERR_CUDA;
    FusedActParams fp;
    GemmParams& p = fp.g;
    p.T = T; p.N = N; p.K = K;
    p.k_blocks_total = K / kBK;
    p.k_splits = 1;
    p.tb8 = 0;
    p.a_scale = nullptr; p.w_scale = w_scale; p.bias = bias;
    p.y = y; p.out_bf16 = (dt == SBN_OUT_BF16);
    p.acc_out = acc_out;
    p.split_acc = nullptr; p.split_counters = nullptr;
    p.w_vals = wvals; p.w_meta = sparse ? meta : nullptr; p.w_tile_bytes = sparse ? 8192 : 16384;
    fp.x_bf16 = x_bf16;
    fp.a_scale_out = a_scale_out;
    const int tiles = (N / kBM) * ((T + 31) / 32);
    const int cluster = pick_cluster_32(sparse, T, N, K);
    cudaError_t err;
    if (sparse) {
        using Cfg = FusedActConfig<true>;
        if (!ensure_dynamic_smem<bitlinear_gemm_fused_act_cluster_kernel<true>>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
        err = launch_kernel_cluster(bitlinear_gemm_fused_act_cluster_kernel<true>, dim3(tiles * cluster), dim3(kSplitThreads),
                                    Cfg::SMEM_BYTES, stream, static_cast<unsigned>(cluster), ta, te, fp);
    } else {
        using Cfg = FusedActConfig<false>;
        if (!ensure_dynamic_smem<bitlinear_gemm_fused_act_cluster_kernel<false>>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
        err = launch_kernel_cluster(bitlinear_gemm_fused_act_cluster_kernel<false>, dim3(tiles * cluster), dim3(kSplitThreads),
                                    Cfg::SMEM_BYTES, stream, static_cast<unsigned>(cluster), ta, te, fp);
    }
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

sbn_status sbn_quant_act_sparse_bitlinear(const void* x_bf16, int T, const int8_t* vals, const uint8_t* meta,
                                          const float* w_scale, int N, int K, const float* bias, void* y,
                                          sbn_out_dtype dt, int32_t* acc_out, float* a_scale_out, void* stream) {
    return run_fused_act(true, x_bf16, T, vals, meta, w_scale, N, K, bias, y, dt, acc_out, a_scale_out,
                         static_cast<cudaStream_t>(stream));
}

sbn_status sbn_quant_act_bitlinear(const void* x_bf16, int T, const int8_t* dense_q, const float* w_scale, int N, int K,
                                   const float* bias, void* y, sbn_out_dtype dt, int32_t* acc_out, float* a_scale_out,
                                   void* stream) {
    return run_fused_act(false, x_bf16, T, dense_q, nullptr, w_scale, N, K, bias, y, dt, acc_out, a_scale_out,
                         static_cast<cudaStream_t>(stream));
}

sbn_status sbn_pack_vals2(const int8_t* vals, int N, int K, uint8_t* vals2, void* stream) {
    if (!vals || !vals2) return SBN_ERR_NULL;
    if (N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (misaligned(vals, 16) || misaligned(vals2, 16)) return SBN_ERR_ALIGN;
    return launch_pack_vals2(vals, N, K, vals2, static_cast<cudaStream_t>(stream));
}

sbn_status sbn_sparse_bitlinear_packed(const int8_t* xq, const float* a_scale, int T, const uint8_t* vals2,
                                       const uint8_t* meta, const float* w_scale, int N, int K, const float* bias,
                                       void* y, sbn_out_dtype dt, int32_t* acc_out, void* stream) {
    if (!xq || !a_scale || !vals2 || !meta || !w_scale || !y) return SBN_ERR_NULL;
    if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (dt != SBN_OUT_F32 && dt != SBN_OUT_BF16) return SBN_ERR_UNSUPPORTED;
    if (T > 1024 || K < 2 * kBK) return SBN_ERR_UNSUPPORTED;          // the few-token regime only
    if (misaligned(xq, 16) || misaligned(vals2, 16) || misaligned(meta, 16) || misaligned(y, 16) || misaligned(a_scale, 4) ||
        misaligned(w_scale, 4) || (acc_out && misaligned(acc_out, 4)) || (bias && misaligned(bias, 4)))
        return SBN_ERR_ALIGN;
    if (use_few_kernel<kFewPacked, false>(T, N, K)) {
        const FewParams p = few_params(T, N, K, xq, nullptr, a_scale, nullptr, vals2, meta, w_scale, bias, y, dt, acc_out);
        return launch_few<kFewPacked, false>(p, static_cast<cudaStream_t>(stream));
    }
    using Cfg = PackedSplitConfig;
    CUtensorMap tb;
    if (!encode_flat_1k(&tb, xq, xq_tiled_bytes(T, K), Cfg::BN / 8)) return SBN_ERR_CUDA;
    GemmParams p;
    p.T = T; p.N = N; p.K = K;
    p.k_blocks_total = K / kBK;
    p.k_splits = 1;
    p.tb8 = static_cast<int>(xq_tb8(T));
    p.a_scale = a_scale; p.w_scale = w_scale; p.bias = bias;
    p.y = y; p.out_bf16 = (dt == SBN_OUT_BF16);
    p.acc_out = acc_out;
    p.split_acc = nullptr; p.split_counters = nullptr;
    p.w_vals = vals2; p.w_meta = meta; p.w_tile_bytes = kVals2TileBytes;
    const int tiles = (N / kBM) * ((T + Cfg::BN - 1) / Cfg::BN);
    const int cluster = pick_cluster_32(true, T, N, K);
    if (!ensure_dynamic_smem<bitlinear_gemm_packed_cluster_kernel>(Cfg::SMEM_BYTES)) return SBN_ERR_CUDA;
    const cudaError_t err = launch_kernel_cluster(bitlinear_gemm_packed_cluster_kernel, dim3(tiles * cluster), dim3(kSplitThreads),
                                                  Cfg::SMEM_BYTES, static_cast<cudaStream_t>(stream), static_cast<unsigned>(cluster), tb, p);
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

static sbn_status canonical_any(bool to_tiled, const void* vals_in, const void* meta_in, int N, int K, void* vals_out,
                                void* meta_out, void* stream) {
    if ((!vals_in) != (!vals_out) || (!meta_in) != (!meta_out) || (!vals_in && !meta_in)) return SBN_ERR_NULL;
    if (N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    if (misaligned(vals_in, 16) || misaligned(vals_out, 16) || misaligned(meta_in, 16) || misaligned(meta_out, 16))
        return SBN_ERR_ALIGN;
    if ((vals_in && vals_in == vals_out) || (meta_in && meta_in == meta_out)) return SBN_ERR_UNSUPPORTED;   // not in place
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return to_tiled ? launch_canonical_layout<true>(vals_in, vals_out, meta_in, meta_out, N, K, s)
                    : launch_canonical_layout<false>(vals_in, vals_out, meta_in, meta_out, N, K, s);
}

sbn_status sbn_unpack_canonical(const int8_t* vals, const uint8_t* meta, int N, int K, int8_t* vals_out,
                                uint8_t* meta_out, void* stream) {
    return canonical_any(false, vals, meta, N, K, vals_out, meta_out, stream);
}

sbn_status sbn_tile_canonical(const int8_t* vals_plain, const uint8_t* meta_plain, int N, int K, int8_t* vals,
                              uint8_t* meta, void* stream) {
    return canonical_any(true, vals_plain, meta_plain, N, K, vals, meta, stream);
}

sbn_status sbn_bitlinear_backward(const void* dY_bf16, int T, const int8_t* xq, const float* a_scale, const int8_t* vals,
                                  const uint8_t* meta, const float* w_scale, int N, int K, void* dX_bf16, float* dW,
                                  void* ws, size_t ws_bytes, void* stream) {
    if (!dY_bf16 || (!dX_bf16 && !dW)) return SBN_ERR_NULL;
    if (dX_bf16 && (!vals || !meta || !w_scale)) return SBN_ERR_NULL;
    if (dW && (!xq || !a_scale)) return SBN_ERR_NULL;
    if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0 || K > (1 << 20)) return SBN_ERR_SHAPE;
    const BackwardWs lay = backward_ws_layout(T, N, K);
    if (!ws || ws_bytes < lay.total) return SBN_ERR_WORKSPACE;
    if (misaligned(dY_bf16, 16) || misaligned(ws, 256) || (dX_bf16 && (misaligned(dX_bf16, 16) || misaligned(vals, 16) || misaligned(meta, 16) || misaligned(w_scale, 4))) ||
        (dW && (misaligned(dW, 16) || misaligned(xq, 16) || misaligned(a_scale, 4))))
        return SBN_ERR_ALIGN;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return run_backward(dY_bf16, T, xq, a_scale, vals, meta, w_scale, N, K, dX_bf16, dW, ws, s);
}

sbn_status sbn_check_status(void* stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return SBN_ERR_CUDA;
    int h = 0;
    if (cudaMemcpyFromSymbol(&h, g_device_status, sizeof(int)) != cudaSuccess) return SBN_ERR_CUDA;
    if (h != 0) {
        const int zero = 0;
        cudaMemcpyToSymbol(g_device_status, &zero, sizeof(int));
        return static_cast<sbn_status>(h);
    }
    return SBN_OK;
}

const char* sbn_status_string(sbn_status s) {
    switch (s) {
        case SBN_OK: return "ok";
        case SBN_ERR_NULL: return "a required pointer is NULL";
        case SBN_ERR_SHAPE: return "bad shape (need T >= 1, N % 128 == 0, K % 128 == 0)";
        case SBN_ERR_ALIGN: return "pointer not 16-byte aligned";
        case SBN_ERR_UNSUPPORTED: return "unsupported pattern, dtype or op";
        case SBN_ERR_WORKSPACE: return "workspace missing or too small";
        case SBN_ERR_CUDA: return "CUDA call failed";
        case SBN_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case SBN_ERR_TOO_LARGE: return "problem larger than the library's built-in scratch can serve";
        default: return "unknown status";
    }
}

void sbn_plan_gemm(int sparse, int T, int N, int K, int* out4) {
    if (!out4) return;
    out4[0] = out4[1] = out4[2] = out4[3] = 0;
    if (T <= 0 || N <= 0 || K <= 0 || N % kBM != 0 || K % kBK != 0) return;
    const GemmPlan g = plan_gemm(sparse != 0, false, T, N, K);
    out4[0] = g.pair ? (g.mt == 1 ? 3 : 2) : (g.cluster > 1 ? 1 : (g.cluster == 1 ? 4 : 0));
    out4[1] = g.bn;
    out4[2] = g.splits;
    out4[3] = g.cluster > 1 ? g.cluster : 0;
}

sbn_status sbn_set_wait_test(int break_waits, unsigned long long wait_limit_us) {
    const unsigned long long ns = wait_limit_us == 0ull ? kWaitLimitNs : wait_limit_us * 1000ull;
    if (cudaMemcpyToSymbol(g_wait_limit_ns, &ns, sizeof(ns)) != cudaSuccess) return SBN_ERR_CUDA;
    g_test_break_waits = break_waits ? 1 : 0;
    return SBN_OK;
}

void sbn_set_gemm_probe(int flags) { g_gemm_probe = flags; }

void sbn_set_gemm_tuning(int token_tile, int split_k) {
    g_force_token_tile = token_tile;
    g_force_split_k = split_k;
}

unsigned long long sbn_launch_count(void) { return g_launch_count.load(); }

}  // extern "C"
