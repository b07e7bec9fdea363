// The two contractions of a layer's backward pass (Sec. 2.3, Eq. 5) in bf16 with fp32 accumulation on the 5th-generation
// tensor cores, in ONE persistent launch:
//
//   part 0   dW [N][K] = dY^T x_q      contraction over the tokens; A = dY [T][N] read MN-major
//   part 1   dX [T][K] = dY W_eff      contraction over the features; A = dY [T][N] read K-major; times bf16(w_scale)
//
// B (x_q [T][K] resp. W_eff [N][K], backward_prep.cuh) is read MN-major in both.  Two CTAs of a cluster issue one
// `tcgen05.mma.cta_group::2.kind::f16` (M = 256: each CTA supplies 128 rows of A and half of the B tile and keeps its
// 128 x BN slice of the accumulator in its own tensor memory).  Operands come by TMA from plain row-major tensors, seven
// stages of 64 contraction steps; the full barrier of a stage lives in the leader CTA and collects both CTAs' bytes,
// `tcgen05.commit ... multicast::cluster` releases stages and publishes accumulators in both CTAs.  The two 256-column
// halves of tensor memory alternate as accumulators, so the epilogue of a tile (a thread owns an output row and writes
// 128 B or 64 B runs of it) runs under the next tile's MMAs.  No TMA multicast.  All waits are bounded.
//
//   warps        0 TMA producer (both CTAs), 1 MMA issuer (leader CTA only; both allocate TMEM),
//                2..9 epilogue: warp w reads TMEM lane quarter w % 4, the even (w < 6) or odd 32-column chunks
//   per stage    A 128 rows x 128 B (16 KB) | B BN/2 rows x 128 B (<= 16 KB): K step of 64 elements, four MMAs of K = 16
//
// Bound by the tensor cores under the power cap: 256 x 256 x 64 takes 0.36 us per pair, 1.7 PFLOP/s while all pairs work.
// Both gradients, preparation included, calls back to back at 4096 tokens (us, two launches with their own waves and
// separate preparation kernels before): 2560 -> 3840 135 -> 119, 2560 -> 2560 110 -> 80, 2560 -> 6912 246 -> 207,
// 6912 -> 2560 234 -> 209.  Converting one operand on spare warps of this kernel, under the other part's tiles, was slower
// (138, 110, 228, 247): the conversion's loads and stores cost the main loop more than the launch they save.
//
// Tiles are 256 x 256, or halves of 256 x 128 where those even out the pairs (backward_plan.h): every pair has a list of
// its own, made so that all end at about the same time although the two parts' tiles differ in length.
#pragma once

#include "backward_plan.h"
#include "gemm_pair_tcgen05.cuh"

namespace sbn {

constexpr int kBf16EpiWarps = 8;
constexpr int kBf16Threads = 32 * (2 + kBf16EpiWarps);
constexpr int kBf16StageA = 128 * 128;                      // bytes
constexpr int kBf16StageB = 128 * 128;                      // bytes reserved (BN/2 <= 128 rows)
constexpr int kBf16StageBytes = kBf16StageA + kBf16StageB;
constexpr int kBf16Stages = 7;
constexpr int kBf16SmemBytes = kBf16Stages * kBf16StageBytes + kBarrierBytes;
static_assert(kBf16SmemBytes <= 232448, "shared memory overflow");

struct Bf16Part {
    int M, Kc;                   // output rows, contraction length
    void* out;                   // [M][K] row-major
    int out_bf16;                // else fp32
    const float* scale;          // device, one fp32, or null: the result is multiplied by bf16(scale)
};
struct Bf16GemmParams {
    Bf16Part part[2];            // dW, dX
    int Nn;                      // output columns of both (K)
    BackwardPlan plan;
};

__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar_cluster_addr) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar_cluster_addr)
        : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Instruction descriptor for kind::f16: D = fp32, A = B = bf16; A K-major or MN-major (bit 15), B MN-major (bit 16).
__host__ __device__ constexpr uint32_t make_idesc_bf16(int mma_m, int mma_n, bool a_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn_major ? (1u << 15) : 0u) | (1u << 16) |
           (static_cast<uint32_t>(mma_n >> 3) << 17) | (static_cast<uint32_t>(mma_m >> 4) << 24);
}

struct Bf16Tile { int part, m0, n0, bn; };
// Entry `i` of this pair in segment `g` (backward_plan.h).
__device__ __forceinline__ Bf16Tile bf16_tile(const Bf16GemmParams& p, int g, int pair, int i) {
    const BackwardSegment& sg = p.plan.seg[g];
    const int u = sg.index(pair, i);
    const int tiles_m = (p.part[sg.part].M + 255) / 256;
    const int tile = sg.half ? sg.first_tile + (u >> 1) : u;
    return Bf16Tile{sg.part, (tile % tiles_m) * 256, (tile / tiles_m) * 256 + (sg.half ? (u & 1) * 128 : 0), sg.half ? 128 : 256};
}

// Tensor maps.  MN-major operands are fetched as 3-D boxes {64 columns, 64 contraction rows, 1 or 2 blocks of 64 columns}:
// a block of 64 rows x 128 B is the MN-major shared-memory image of 64 output rows (or columns) -- 8-row groups 1 KB apart
// along the contraction (the stride offset), blocks 8 KB apart (the leading offset); an MMA of K = 16 starts 2 KB further per
// step.  One instruction per operand and stage: TMA takes about 64 ns per instruction and 2.8 ns per KB, so that with one
// instruction per block (four per stage) the loads, 0.35 us per stage, paced the loop, not the MMAs (0.28).
struct Bf16Maps {
    CUtensorMap aw;              // dY [T][N] for dW: two blocks
    CUtensorMap ax;              // dY [T][N] for dX: K-major, box {64 of N, 128 tokens}
    CUtensorMap b[2][2];         // x_q [T][K], W_eff [N][K]: two blocks, one block (half tiles)
};
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kBf16Threads, 1)
backward_gemm_kernel(const __grid_constant__ Bf16Maps maps, const __grid_constant__ Bf16GemmParams p) {
    constexpr int STAGES = kBf16Stages;

    pdl_launch_dependents();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = smem_u32(smem_raw);
    if (smem_base & 1023u) {          // swizzled tiles need 1 KB alignment; identical in every CTA
        if (threadIdx.x == 0) atomicExch(&g_device_status, static_cast<int>(SBN_ERR_CUDA));
        return;
    }
    const uint32_t bar_base = smem_base + STAGES * kBf16StageBytes;
    const uint32_t bar_full = bar_base;
    const uint32_t bar_empty = bar_full + 8 * STAGES;
    const uint32_t bar_acc_full = bar_empty + 8 * STAGES;     // [2]
    const uint32_t bar_acc_empty = bar_acc_full + 16;         // [2]
    const uint32_t tmem_slot = bar_acc_empty + 16;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + (tmem_slot + 8 - smem_base));

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair_id = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_acc_full + 8 * i, 1);
            mbar_init(bar_acc_empty + 8 * i, 2 * kBf16EpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, kTmemCols);
        tcgen05_fence_before();
    }
    __syncthreads();
    cluster_sync_all();
    tcgen05_fence_after();
    pdl_wait();                       // nothing above touches global memory
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int g = 0; ok && g < p.plan.segments; ++g) {
                for (int i = 0; ok && i < p.plan.seg[g].count(pair_id); ++i) {
                    const Bf16Tile t = bf16_tile(p, g, pair_id, i);
                    const int half_bn = t.bn >> 1;
                    const uint32_t bytes_per_cta = static_cast<uint32_t>(kBf16StageA + half_bn * 128);
                    const int m0 = t.m0 + static_cast<int>(rank) * 128;
                    const int n0 = t.n0 + static_cast<int>(rank) * half_bn;
                    const int k_stages = (p.part[t.part].Kc + 63) / 64;
                    const CUtensorMap* tb = &maps.b[t.part][t.bn == 128];
                    for (int ks = 0; ks < k_stages; ++ks) {
                        if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
                        const uint32_t full_leader = map_to_cta(bar_full + 8 * stage, 0);
                        if (rank == 0) mbar_expect_tx(bar_full + 8 * stage, 2 * bytes_per_cta);
                        const uint32_t st = smem_base + stage * kBf16StageBytes;
                        // rows or columns beyond the tensors are zero-filled by the hardware and still count their full size
                        if (t.part == 0) {
                            tma_load_3d_pair(st, &maps.aw, 0, ks * 64, m0 >> 6, full_leader);
                        } else {
                            tma_load_2d_pair(st, &maps.ax, ks * 64, m0, full_leader);
                        }
                        tma_load_3d_pair(st + kBf16StageA, tb, 0, ks * 64, n0 >> 6, full_leader);
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (leader)
        if (rank == 0 && lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t acc_iter = 0;
            bool ok = true;
            for (int g = 0; ok && g < p.plan.segments; ++g) {
                const int part = p.plan.seg[g].part;
                const uint32_t idesc = make_idesc_bf16(256, p.plan.seg[g].half ? 128 : 256, part == 0);
                const int k_stages = (p.part[part].Kc + 63) / 64;
                // K = 16 elements per instruction: 16 rows of an MN-major operand, 32 B along a row of a K-major one
                const uint64_t a_step = part == 0 ? (2048 >> 4) : (32 >> 4);
                const uint32_t a_lbo = part == 0 ? 8192 : 16;
                for (int i = 0; ok && i < p.plan.seg[g].count(pair_id); ++i) {
                    const uint32_t buf = acc_iter & 1u;
                    const uint32_t acc_phase = (acc_iter >> 1) & 1u;
                    if (!mbar_wait(bar_acc_empty + 8 * buf, acc_phase ^ 1u, abort_flag)) { ok = false; break; }
                    tcgen05_fence_after();
                    const uint32_t d_tmem = tmem_base + buf * 256u;
                    for (int ks = 0; ks < k_stages; ++ks) {
                        if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag)) { ok = false; break; }
                        tcgen05_fence_after();
                        const uint32_t st = smem_base + stage * kBf16StageBytes;
                        const uint64_t a_desc = make_smem_desc(st, a_lbo, 1024, kSwz128);
                        const uint64_t b_desc = make_smem_desc(st + kBf16StageA, 8192, 1024, kSwz128);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            mma_bf16_pair(d_tmem, a_desc + a_step * q, b_desc + (2048u >> 4) * q, idesc, (ks | q) != 0 ? 1u : 0u);
                        tcgen05_commit_pair(bar_empty + 8 * stage);
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (!ok) break;
                    tcgen05_commit_pair(bar_acc_full + 8 * buf);
                    ++acc_iter;
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (8 warps)
        const int quarter = warp & 3;                     // TMEM lane quarter this warp may read
        const int parity = (warp - 2) >> 2;               // even or odd 32-column chunks
        const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
        uint32_t acc_iter = 0;
        bool ok = true;
        for (int g = 0; ok && g < p.plan.segments; ++g) {
            const Bf16Part& pt = p.part[p.plan.seg[g].part];
            float scale = 1.0f;
            if (pt.scale != nullptr) scale = __uint_as_float(f32_to_bf16_rne(__ldg(pt.scale)) << 16);    // the scale as a bf16 run holds it
            for (int i = 0; i < p.plan.seg[g].count(pair_id); ++i) {
                const Bf16Tile t = bf16_tile(p, g, pair_id, i);
                const int m = t.m0 + static_cast<int>(rank) * 128 + quarter * 32 + lane;
                const uint32_t buf = acc_iter & 1u;
                const uint32_t acc_phase = (acc_iter >> 1) & 1u;
                const uint32_t acc_empty_leader = map_to_cta(bar_acc_empty + 8 * buf, 0);
                if (!mbar_wait(bar_acc_full + 8 * buf, acc_phase, abort_flag)) { ok = false; break; }
                tcgen05_fence_after();
                const uint32_t t_addr = tmem_base + lane_base + buf * 256u;
                const int chunks = t.bn >> 5;
#pragma unroll 1
                for (int c = parity; c < chunks; c += 2) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t r[16];
                        tmem_ld_32x32b_x16(t_addr + static_cast<uint32_t>(c * 32 + h * 16), r);
                        tmem_ld_wait();
                        if (c + 2 >= chunks && h == 1) {
                            tcgen05_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive_cluster(acc_empty_leader);
                        }
                        const int n = t.n0 + c * 32 + h * 16;
                        if (m < pt.M && n < p.Nn) {       // Nn % 16 == 0: a run of 16 columns is in or out as a whole
                            if (pt.out_bf16) {
                                uint32_t pk[8];
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const float v0 = __fmul_rn(__uint_as_float(r[2 * j]), scale), v1 = __fmul_rn(__uint_as_float(r[2 * j + 1]), scale);
                                    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(v1), "f"(v0));
                                }
                                uint4* o = reinterpret_cast<uint4*>(static_cast<uint16_t*>(pt.out) + static_cast<size_t>(m) * p.Nn + n);
                                o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                                o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                            } else {
                                float4* o = reinterpret_cast<float4*>(static_cast<float*>(pt.out) + static_cast<size_t>(m) * p.Nn + n);
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    o[j] = make_float4(__fmul_rn(__uint_as_float(r[4 * j]), scale), __fmul_rn(__uint_as_float(r[4 * j + 1]), scale),
                                                       __fmul_rn(__uint_as_float(r[4 * j + 2]), scale), __fmul_rn(__uint_as_float(r[4 * j + 3]), scale));
                            }
                        }
                    }
                }
                ++acc_iter;
            }
        }
    }

    // teardown: nobody leaves while the peer may still touch this CTA's smem, barriers or TMEM
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        __syncwarp();
        tcgen05_fence_after();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace sbn
