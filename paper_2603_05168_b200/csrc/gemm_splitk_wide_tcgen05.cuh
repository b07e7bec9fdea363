// Eq. 4 for a few hundred tokens: split-K inside a thread-block cluster, with the whole chunk of tokens in one tile.
//
// From about a hundred tokens on a 128-feature tile that walks all of K is paced by the instructions of its K-loop
// (0.23 us per 128 columns whatever its token width up to 128), so narrow token tiles repeat that walk for the same
// weights, and the reduce-scatter of gemm_splitk_cluster_tcgen05.cuh, one 4-byte store per partial sum, costs more
// than the K-loop it saves (0.02 to 0.03 us per token).  Here a tile has up to 256 tokens (runtime width, a multiple of
// 16) -- every weight is read by one cluster -- the S CTAs of a cluster split its K-blocks evenly, and the partial
// sums travel as bulk copies:
//
//   warp 0        TMA producer (weights of the first stages before the dependency wait), warp 1 MMA issuer
//   epilogue      8 warps copy the accumulator into P [token][128 features] int32, which takes the place of the
//                 pipeline stages; CTA r owns the tokens [r c, (r+1) c) of the tile, c = ceil(tokens / S)
//   exchange      one cp.async.bulk per peer sends that peer's tokens into its slot of the receive area, which counts
//                 the bytes on an mbarrier of the receiver.  Both areas lie where the stages were, so nobody sends
//                 before every CTA of the cluster has reported its last MMA (bar_ready)
//   finish        own partials + S - 1 slots, dequantised (+ bias), stored; a warp stores 32 features of a token
//
// Measured (time stamps, 2560 -> 3840, 201 tokens in two tiles of 112, S = 2, 120 CTAs): dependency wait to last MMA 3.0 us
// for 10 K-blocks (one per stage), peers' half of P 0.3, exchange 0.75, finish 0.5; chained with the quantiser 8.4 us, against
// 10.3 unsplit in 64-token tiles and 9.9 with one store per partial sum.  What the exchange costs is per token and peer:
// 0.03 us x tokens x (S - 1) / S, mostly the copies between the SMs (about 38 GB/s each way per SM), so S stays at 2 to 4.
// 6912 -> 2560 at 201 tokens 14.4 -> 10.6, 11008 -> 4096 21.3 -> 16.2; dense at 512 tokens 22.4 -> 17.6 and 38.4 -> 26.8.
//
// No CTA leaves before all have received everything (cluster barrier): the sources of the copies stay in place.  All
// mbarrier waits are bounded.
#pragma once

#include "gemm_splitk_cluster_tcgen05.cuh"

namespace sbn {

constexpr int kWideEpiWarps = 8;
constexpr int kWideThreads = 32 * (2 + kWideEpiWarps);
constexpr int kWideMaxStages = 8;
constexpr int kWideMinBn = 80;                              // narrower tiles belong to the narrow-tile kernel
constexpr int kWideDataBytes = 224 * 1024;                  // stages, then P and the receive area
constexpr int kWideSmemBytes = 1024 + kWideDataBytes + kBarrierBytes;
static_assert(kWideSmemBytes + 1024 + 64 <= 232448, "shared memory overflow");
// A CTA of the activation quantiser (1 KB that the system takes, 128 B) fits beside one of these to the byte: in a chain of quantisers
// and GEMMs the next quantiser is then resident before this kernel ends.  With 512 B more here every such GEMM took 0.4 to
// 0.7 us longer (dense 2560 -> 2560, 256 tokens 8.5 / 9.2; 2560 -> 3840 9.3 / 9.7; 6912 -> 2560 sparse, 201 tokens 10.6 / 10.9).
constexpr int kWideStaticSmemBytes = 640;                   // what ptxas reports for this kernel
static_assert(kWideSmemBytes + kWideStaticSmemBytes + 1024 + (1024 + 128) <= 228 * 1024, "the quantiser no longer fits beside");
constexpr uint32_t kWideTmemCols = 512;                     // accumulator up to 256, metadata above it
constexpr int kWideMetaCol0 = 256;

__host__ __device__ constexpr int wide_block_bytes(bool sparse, int bn) { return (sparse ? kBM * (kBK / 2 + kBK / 8) : kBM * kBK) + bn * kBK; }
// K-blocks per stage.  TMA takes about 64 ns per instruction and 2.8 ns per KB, so a stage has two blocks fetched with one
// instruction per operand -- where three such stages fit (sparse up to 208 tokens, dense up to 160).  Quantiser + GEMM, us,
// one block / two: 6912 -> 2560 256 tokens in tiles of 128 13.1 / 11.7, 4096 -> 4096 11.9 / 10.5, 11008 -> 4096 201 tokens in
// one tile 17.1 / 16.2; with room for two stages of two only, tiles of 256 19.0 / 20.3, dense tiles of 208 24.0 / 27.5.
__host__ __device__ constexpr int wide_group(bool sparse, int bn) { return 6 * wide_block_bytes(sparse, bn) <= kWideDataBytes ? 2 : 1; }
// Does the exchange fit (P and S - 1 slots of ceil(bn / S) tokens, 512 B per token)?
__host__ __device__ constexpr bool wide_fits(int bn, int S) { return (bn + (S - 1) * ((bn + S - 1) / S)) * kBM * 4 <= kWideDataBytes; }

__device__ __forceinline__ void bulk_copy_to_cta(uint32_t dst_cluster, uint32_t src_cta, uint32_t bytes, uint32_t bar_cluster) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_cluster), "r"(src_cta), "r"(bytes), "r"(bar_cluster) : "memory");
}

// tmap_a / tmap_e: weight tiles and metadata as rows of 1 KB, boxes of G tiles; tmap_b: xq as rows of 1 KB, box of bn / 8
// (G = 1), or as [K / 128][atoms][1 KB], box of 2 x bn / 8 atoms.  A stage holds G = wide_group K-blocks: weights of all, metadata of all, activations of all.  The
// second block of a slice of odd length is loaded and not used (beyond the arrays the hardware fills in zeros).
template <bool SPARSE, int G>
__global__ void __launch_bounds__(kWideThreads, 1)
bitlinear_gemm_splitk_wide_kernel(const __grid_constant__ CUtensorMap tmap_a,
                                  const __grid_constant__ CUtensorMap tmap_b,
                                  const __grid_constant__ CUtensorMap tmap_e,
                                  const GemmParams p, const int bn) {
    constexpr int A_BYTES = SPARSE ? kBM * (kBK / 2) : kBM * kBK;
    constexpr int E_BYTES = SPARSE ? kBM * (kBK / 8) : 0;
    const int stage_bytes = G * wide_block_bytes(SPARSE, bn);
    const int stages = min(kWideMaxStages, kWideDataBytes / stage_bytes);

    extern __shared__ uint8_t smem_raw[];
    // 1 KB alignment for the 128 B swizzle atoms; the offset is the same in every CTA of the cluster
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar_full = smem_base + kWideDataBytes;
    const uint32_t bar_empty = bar_full + 8 * kWideMaxStages;
    const uint32_t bar_acc_full = bar_empty + 8 * kWideMaxStages;
    const uint32_t bar_ready = bar_acc_full + 8;             // every CTA of the cluster has finished its MMAs
    const uint32_t bar_recv = bar_ready + 8;                 // counts the bytes of partial sums sent to this CTA
    const uint32_t tmem_slot = bar_recv + 8;

    __shared__ int s_abort;
    __shared__ float s_scale_split[128];                     // of the tokens this CTA finishes, S > 1 (at most 128 then)
    volatile int* abort_flag = &s_abort;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int rank = static_cast<int>(cluster_ctarank());
    const int S = static_cast<int>(cluster_nctarank());
    const int tile = blockIdx.x / S;                         // clusters are consecutive blocks
    const int tiles_m = p.N / kBM;
    const int mt = tile % tiles_m;
    const int t0 = (tile / tiles_m) * bn;
    const int kb0 = p.k_blocks_total * rank / S;             // never empty: S <= K / 128
    const int kb1 = p.k_blocks_total * (rank + 1) / S;
    const int tokens = min(bn, p.T - t0);                    // real tokens of this tile
    const int share = (tokens + S - 1) / S;
    const int my0 = min(tokens, rank * share);
    const int my_tokens = min(share, tokens - my0);

    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < stages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        mbar_init(bar_acc_full, 1);
        mbar_init(bar_ready, static_cast<uint32_t>(S));
        mbar_init(bar_recv, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar_recv, static_cast<uint32_t>(my_tokens) * static_cast<uint32_t>(S - 1) * (kBM * 4));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kWideTmemCols);
        tcgen05_fence_before();
    }
    __syncthreads();
    tcgen05_fence_after();
    cluster_arrive();                                        // peers' barriers are touched after the matching wait only
    // The weights of the first stages before the dependency wait: no kernel that writes packed weights signals its
    // dependents early (sbn_common.cuh).
    const int n_stages = (kb1 - kb0 + G - 1) / G;                // of this CTA's slice
    const int n_pre = min(stages, n_stages);
    auto load_weights = [&](int stage, int kb) {             // blocks kb .. kb + G - 1
        const uint32_t full = bar_full + 8 * stage;
        const uint32_t st = smem_base + stage * stage_bytes;
        const int wt = mt * p.k_blocks_total + kb;
        mbar_expect_tx(full, static_cast<uint32_t>(stage_bytes));
        if constexpr (SPARSE) {
            tma_load_2d(st, &tmap_a, 0, wt * 8, full);
            tma_load_2d(st + G * A_BYTES, &tmap_e, 0, wt * 2, full);
        } else {
            tma_load_2d(st, &tmap_a, 0, wt * 16, full);
        }
    };
    if (threadIdx.x == 0) {
        tma_prefetch_desc(&tmap_a);
        tma_prefetch_desc(&tmap_b);
        if constexpr (SPARSE) tma_prefetch_desc(&tmap_e);
        for (int i = 0; i < n_pre; ++i) load_weights(i, kb0 + G * i);
        const int rest = kb1 - kb0 - G * n_pre;              // the rest of the slice goes to L2
        if (rest > 0) {
            const size_t wt0 = static_cast<size_t>(mt) * p.k_blocks_total + kb0 + G * n_pre;
            prefetch_l2_bulk(static_cast<const char*>(p.w_vals) + wt0 * p.w_tile_bytes, static_cast<uint32_t>(rest * p.w_tile_bytes));
            if (p.w_meta) prefetch_l2_bulk(static_cast<const char*>(p.w_meta) + wt0 * 2048, static_cast<uint32_t>(rest * 2048));
        }
    }
    pdl_wait();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0 && !p.test_skip_loads) {
            int stage = 0;
            uint32_t phase = 0;
            for (int i = 0; i < n_stages; ++i) {
                if (i >= n_pre) {
                    if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag)) break;
                    load_weights(stage, kb0 + G * i);
                }
                const uint32_t b_dst = smem_base + stage * stage_bytes + G * (A_BYTES + E_BYTES);
                if constexpr (G == 1) tma_load_2d(b_dst, &tmap_b, 0, (kb0 + i) * p.tb8 + (t0 >> 3), bar_full + 8 * stage);
                else tma_load_3d(b_dst, &tmap_b, 0, t0 >> 3, kb0 + G * i, bar_full + 8 * stage);
                if (++stage == stages) { stage = 0; phase ^= 1u; }
            }
        }
        __syncwarp();
        cluster_wait();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = make_idesc_i8(kBM, bn, SPARSE);
            int stage = 0;
            uint32_t phase = 0;
            bool good = true;
            for (int kb = kb0; kb < kb1; kb += G) {
                if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag)) { good = false; break; }
                tcgen05_fence_after();
                const uint32_t st = smem_base + stage * stage_bytes;
                if constexpr (SPARSE) {                          // one copy for both blocks of a stage (see the narrow-tile kernel)
                    const uint32_t e_tmem = tmem_base + static_cast<uint32_t>(kWideMetaCol0 + 8 * stage);
                    if constexpr (G == 2) tcgen05_cp_128x256b(e_tmem, make_smem_desc(st + G * A_BYTES, E_BYTES, 128, kSwzNone));
                    else tcgen05_cp_128x128b(e_tmem, make_smem_desc(st + G * A_BYTES, 128, 128, kSwzNone));
                }
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    if (h > 0 && kb + h >= kb1) break;
                    const uint32_t a_addr = st + h * A_BYTES;
                    const uint32_t b_addr = st + G * (A_BYTES + E_BYTES) + h * bn * kBK;
                    const uint32_t first = (kb + h == kb0) ? 0u : 1u;
                    const uint64_t b_desc = make_smem_desc(b_addr, 16, 1024, kSwz128);
                    if constexpr (SPARSE) {
                        const uint32_t e_tmem = tmem_base + static_cast<uint32_t>(kWideMetaCol0 + 8 * stage + 4 * h);
                        const uint64_t a_desc = make_smem_desc(a_addr, 16, 512, kSwz64);
#pragma unroll
                        for (int j = 0; j < kBK / 64; ++j)
                            mma_i8_sparse(tmem_base, a_desc + static_cast<uint64_t>(2 * j), b_desc + static_cast<uint64_t>(4 * j),
                                          e_tmem + 2 * j, idesc, j == 0 ? first : 1u);
                    } else {
                        const uint64_t a_desc = make_smem_desc(a_addr, 16, 1024, kSwz128);
#pragma unroll
                        for (int j = 0; j < kBK / 32; ++j)
                            mma_i8_dense(tmem_base, a_desc + static_cast<uint64_t>(2 * j), b_desc + static_cast<uint64_t>(2 * j),
                                         idesc, j == 0 ? first : 1u);
                    }
                }
                tcgen05_commit(bar_empty + 8 * stage);
                if (++stage == stages) { stage = 0; phase ^= 1u; }
            }
            if (good) tcgen05_commit(bar_acc_full);
        }
        __syncwarp();
        cluster_wait();
    } else {
        // ------------------------------------------------------------------ epilogue
        const int e = threadIdx.x - 64;                      // 0..255
        const int quarter = warp & 3;                        // TMEM lane quarter this warp may read
        const int half = (warp - 2) >> 2;                    // even or odd 32-column chunks, later even or odd tokens
        const int f = quarter * 32 + lane;                   // feature inside the tile
        const int n4 = mt * kBM + 4 * lane;                  // the finishing loop: four features per thread, a token per warp
        float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (p.bias) {
#pragma unroll
            for (int j = 0; j < 4; ++j) bias[j] = __ldg(p.bias + n4 + j);
        }
        // unsplit: up to 256 scales, at the end of the area that the stages leave once the MMAs are done (P needs at most 128 KB of it)
        float* const s_scale = S == 1 ? reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)) + kWideDataBytes) - 256 : s_scale_split;
        const float scale = e < my_tokens ? __fmul_rn(__ldg(p.w_scale), __ldg(p.a_scale + t0 + my0 + e)) : 0.0f;
        if (S > 1 && e < my_tokens) s_scale[e] = scale;
        bool ok = mbar_wait(bar_acc_full, 0u, abort_flag);
        if (S == 1 && ok) s_scale[e] = scale;
        tcgen05_fence_after();
        cluster_wait();                                      // all peers have started, their barriers exist
        if (ok && e < S) mbar_arrive_cluster(map_to_cta(bar_ready, static_cast<uint32_t>(e)));
        // P [token][128]: where the stages were -- this CTA's MMAs have read them.  The peers' tokens first; this CTA's own
        // while those are under way.
        uint32_t* const P = reinterpret_cast<uint32_t*>(smem_raw + (smem_base - smem_u32(smem_raw)));
        auto put = [&](bool own) {
#pragma unroll 1
            for (int c = half; c * 32 < tokens; c += 2) {
                const bool any_own = c * 32 < my0 + my_tokens && c * 32 + 32 > my0;
                const bool any_other = c * 32 < my0 || min(tokens, c * 32 + 32) > my0 + my_tokens;
                if (own ? !any_own : !any_other) continue;
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(c * 32), r);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int t = c * 32 + j;
                    if (t < tokens && (static_cast<unsigned>(t - my0) < static_cast<unsigned>(my_tokens)) == own) P[t * kBM + f] = r[j];
                }
            }
        };
        if (ok) put(false);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (e < S && e != rank && ok) {                      // thread e sends peer e its tokens
            const int first_tok = min(tokens, e * share);
            const int cnt = min(share, tokens - first_tok);
            if (cnt > 0 && mbar_wait(bar_ready, 0u, abort_flag)) {
                const int slot = rank < e ? rank : rank - 1;
                const uint32_t recv = smem_base + static_cast<uint32_t>((tokens + slot * share) * (kBM * 4));
                bulk_copy_to_cta(map_to_cta(recv, static_cast<uint32_t>(e)), smem_base + static_cast<uint32_t>(first_tok * (kBM * 4)),
                                 static_cast<uint32_t>(cnt * (kBM * 4)), map_to_cta(bar_recv, static_cast<uint32_t>(e)));
            }
        }
        __syncwarp();
        if (ok) put(true);
        tcgen05_fence_before();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (!mbar_wait(bar_recv, 0u, abort_flag)) ok = false;
        const int n_tok = (ok && *abort_flag == 0) ? my_tokens : 0;
        const int4* const mine = reinterpret_cast<const int4*>(P + my0 * kBM) + lane;
        const int4* const recv = reinterpret_cast<const int4*>(P + tokens * kBM) + lane;
        auto finish = [&](auto s_const) {
            constexpr int SS = decltype(s_const)::value;     // 0: run-time S
            const int parts = (SS ? SS : S) - 1;
#pragma unroll 4
            for (int l = warp - 2; l < n_tok; l += kWideEpiWarps) {
                int4 acc = mine[l * (kBM / 4)];
#pragma unroll
                for (int s = 0; s < parts; ++s) {
                    const int4 v = recv[(s * share + l) * (kBM / 4)];
                    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
                }
                const size_t o = static_cast<size_t>(t0 + my0 + l) * p.N + n4;
                if (p.acc_out) { p.acc_out[o] = acc.x; p.acc_out[o + 1] = acc.y; p.acc_out[o + 2] = acc.z; p.acc_out[o + 3] = acc.w; }
                const float sc = s_scale[l];
                float v0 = __fmul_rn(static_cast<float>(acc.x), sc), v1 = __fmul_rn(static_cast<float>(acc.y), sc);
                float v2 = __fmul_rn(static_cast<float>(acc.z), sc), v3 = __fmul_rn(static_cast<float>(acc.w), sc);
                if (p.bias) { v0 = __fadd_rn(v0, bias[0]); v1 = __fadd_rn(v1, bias[1]); v2 = __fadd_rn(v2, bias[2]); v3 = __fadd_rn(v3, bias[3]); }
                if (p.out_bf16)
                    *reinterpret_cast<uint2*>(static_cast<uint16_t*>(p.y) + o) = make_uint2(f32_to_bf16_rne(v0) | (f32_to_bf16_rne(v1) << 16),
                                                                                            f32_to_bf16_rne(v2) | (f32_to_bf16_rne(v3) << 16));
                else
                    *reinterpret_cast<float4*>(static_cast<float*>(p.y) + o) = make_float4(v0, v1, v2, v3);
            }
        };
        if (S == 1) finish(std::integral_constant<int, 1>{});
        else if (S == 2) finish(std::integral_constant<int, 2>{});
        else if (S == 3) finish(std::integral_constant<int, 3>{});
        else if (S == 4) finish(std::integral_constant<int, 4>{});
        else finish(std::integral_constant<int, 0>{});
        __syncwarp();
    }
    // The copies this CTA sent have arrived when every CTA has received its own.
    tcgen05_fence_before();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    cluster_wait();
    if (warp == 1) {
        __syncwarp();
        tcgen05_fence_after();
        tmem_dealloc(tmem_base, kWideTmemCols);
    }
}

}  // namespace sbn
