// Eq. 4 for few tokens: warp-level matrix instructions fed from registers.
//
// With a handful of tokens a BitLinear is a stream over the weights, and what a call costs is a chain of latencies
// around it.  The 5th-generation tensor core is the wrong tool there: a tcgen05.mma into a tile of 32 tokens takes
// as long as one into 240 (65 ns measured, plus a metadata copy per 128 columns), it wants its operands in shared
// memory, its result comes back through tensor memory, and its 128-row tiles have to be split along K over a cluster
// to use all SMs.  A warp-level sparse instruction (m16n8k64) takes 9 clocks per SM quarter, reads both operands from
// registers and needs a tile of 16 features only, so that
//
//   a CTA   owns 16 output features and all of K (and further groups of 16, if there are more groups than CTAs); its
//           warps take the 128-column blocks in turn and add their partial sums through shared memory: no cluster, no
//           tensor memory, no barrier before the last one;
//   a warp  loads the weights of its first blocks into registers BEFORE the dependency wait (they do not
//           depend on the kernel before; see sbn_common.cuh for why that is safe), straight from the tiled
//           layout and coalesced: of a 16-row, 128-column block a lane takes one 16-byte piece of each of two rows
//           and one row's metadata;
//   tokens  8 per instruction, NT (1 or 2) groups of 8 per CTA; the activations of a block are two 16-byte loads per lane
//           and group, right from the tiled layout.
//
// Nothing is staged or shuffled because the order of K inside a block is free as long as both operands agree.  With
// g = lane / 4, q = lane % 4: of a row's 128 columns the activation side reads chunks q and 4 + q (16 columns each), the
// weight side columns 32 q .. 32 q + 31; which of them meet at a contraction index is said at the operand words below.
// (Weights through a cp.async ring in shared memory instead of registers were tried: 0.2 to 0.6 us slower.)
//
// Three weight forms: dense int8, 2:4 values + metadata, 2:4 values packed at two bits + metadata.  FUSED: the
// activations arrive as bf16 and every CTA quantises them itself (Sec. 2.1; it sees all of K, so a token's
// maximum needs one exchange through shared memory); saves the quantiser's launch, costs reading bf16 twice in every CTA.
#pragma once

#include "gemm_tcgen05.cuh"
#include "quant_act.cuh"

namespace sbn {

enum FewWeights { kFewDense = 0, kFewSparse = 1, kFewPacked = 2 };

struct FewParams {
    int T, N, k_blocks;              // k_blocks = K / 128
    int tb8;                         // 8-token atoms per block of the tiled xq (2 * ceil(T / 16))
    const uint8_t* xq;               // tiled int8 activations, or
    const uint4* x_bf16;             // (FUSED) bf16 [T][K]
    const float* a_scale;            // [T] (not FUSED)
    float* a_scale_out;              // [T] or null (FUSED)
    const uint8_t* vals;             // dense_q, vals or vals2, tiled
    const uint8_t* meta;             // tiled (not dense)
    const float* w_scale;
    const float* bias;               // [N] or null
    void* y;                         // [T][N] fp32 or bf16
    int out_bf16;
    int32_t* acc_out;                // [T][N] or null
};

__device__ __forceinline__ void mma_m16n8k64_sp(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3, uint32_t e) {
    asm volatile(
        "mma.sp::ordered_metadata.sync.aligned.m16n8k64.row.col.s32.s8.s8.s32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9, %10, %11}, {%0, %1, %2, %3}, %12, 0x0;"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(b2), "r"(b3), "r"(e));
}
__device__ __forceinline__ void mma_m16n8k32(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// A lane's weights of one 16-row x 128-column block, as loaded.
template <int WT> struct FewBlock;
template <> struct FewBlock<kFewDense> { uint4 w[2][2]; };                   // [row g, g + 8][chunk q, 4 + q]
template <> struct FewBlock<kFewSparse> { uint4 w[2]; uint4 m; };            // values of rows g, g + 8; metadata of row g + 8 (lane & 1)
template <> struct FewBlock<kFewPacked> { uint32_t w[2]; uint4 m; };

// Weights are read once: they leave L1 alone.
__device__ __forceinline__ uint4 ldg_once(const uint8_t* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t ldg_once_u32(const uint8_t* p) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// The warp's loads: blocks kb = warp, warp + W, ... of row groups blockIdx.x, + gridDim.x, ...  16 rows are contiguous in
// every layout (1 KB of values, 256 B of metadata, 2 KB of dense weights) and repeat its swizzle.
template <int WT, int W>
struct FewFetch {
    const uint8_t *w, *w2, *m;       // this lane's next pieces (w2: dense, the second chunk)
    int group, n_groups, kb, k_blocks, rounds_end;
    __device__ __forceinline__ FewFetch(const FewParams& p, uint32_t lane, int warp, int rounds)
        : w2(nullptr), m(nullptr), group(blockIdx.x), n_groups(p.N >> 4), kb(warp), k_blocks(p.k_blocks), rounds_end(rounds * W) { place(p, lane); }
    __device__ __forceinline__ void place(const FewParams& p, uint32_t lane) {
        const uint32_t g = lane >> 2, q = lane & 3u, sub = group & 7u;
        const size_t tile = static_cast<size_t>(group >> 3) * k_blocks + kb;
        if constexpr (WT == kFewDense) {
            w = p.vals + tile * 16384 + sub * 2048u + sw128_in_tile(g, 16u * q);
            w2 = p.vals + tile * 16384 + sub * 2048u + sw128_in_tile(g, 64u + 16u * q);
        } else {
            w = WT == kFewSparse ? p.vals + tile * 8192 + sub * 1024u + vals_in_tile(g, 16u * q) : p.vals + tile * 2048 + sub * 256u + g * 16u + 4u * q;
            m = p.meta + tile * 2048 + sub * 256u + (g + 8u * (lane & 1u)) * 16u;
        }
    }
    __device__ __forceinline__ void next(const FewParams& p, uint32_t lane, FewBlock<WT>& b) {
        if (group < n_groups && kb < k_blocks) {
            if constexpr (WT == kFewDense) {
                b.w[0][0] = ldg_once(w);
                b.w[0][1] = ldg_once(w2);
                b.w[1][0] = ldg_once(w + 1024);
                b.w[1][1] = ldg_once(w2 + 1024);
            } else if constexpr (WT == kFewSparse) {
                b.w[0] = ldg_once(w);
                b.w[1] = ldg_once(w + 512);
                b.m = ldg_once(m);
            } else {
                b.w[0] = ldg_once_u32(w);
                b.w[1] = ldg_once_u32(w + 128);
                b.m = ldg_once(m);
            }
        }
        kb += W;
        constexpr size_t kStep = static_cast<size_t>(W) * (WT == kFewDense ? 16384 : (WT == kFewSparse ? 8192 : 2048));
        w += kStep;
        if constexpr (WT == kFewDense) w2 += kStep; else m += static_cast<size_t>(W) * 2048;
        if (kb >= rounds_end) {                                              // next row group
            kb -= rounds_end;
            group += gridDim.x;
            place(p, lane);
        }
    }
};

// The warp's next D blocks go to the L2 before the dependency wait (a lane per block): loaded after it, from memory, they were
// another trip on the critical path.  Quantiser + GEMM in a decode loop, us, without / with: 6912 -> 2560 (seven blocks per warp, four
// in registers) 1 token 6.05 / 5.77, dense 7.2 / 6.6; 4096 -> 11008 (two row groups per CTA) 8.25 / 8.15, dense 9.7 / 9.4.  All of the rest
// at once is too much where memory is the limit (4096 -> 11008 8.5, dense 10.2), and very long rows lose by any of it (11008 -> 4096:
// eleven blocks, 9.37 / 9.45 at 8 tokens, dense 11.5 / 11.7) -- unless they are packed and the memory has time (9.4 / 8.5).  Packed weights gain
// a tenth everywhere, also where there is nothing to prefetch (2560 -> 2560 4.6 / 4.2): without a side effect here the compiler
// expands the first blocks before it asks for the activations.  (It does so too behind an empty asm that takes the blocks' registers
// after the activations' loads: 2560 -> 2560 4.4, 4096 -> 4096 5.2 / 4.4.)
template <int WT, int W, int D>
__device__ __forceinline__ void few_prefetch_next(const FewParams& p, uint32_t lane, uint32_t warp, uint32_t rounds) {
    if (lane >= D || (WT != kFewPacked && rounds > 2 * D)) return;
    const uint32_t i = D + lane, nth = i / rounds, kb = warp + (i - nth * rounds) * W, group = blockIdx.x + nth * gridDim.x;
    if (group >= static_cast<uint32_t>(p.N >> 4) || kb >= static_cast<uint32_t>(p.k_blocks)) return;
    const size_t tile = static_cast<size_t>(group >> 3) * p.k_blocks + kb;
    constexpr uint32_t kRows = WT == kFewDense ? 2048u : (WT == kFewSparse ? 1024u : 256u);       // bytes of 16 rows
    prefetch_l2_bulk(p.vals + tile * (8u * kRows) + (group & 7u) * kRows, kRows);
    if constexpr (WT != kFewDense) prefetch_l2_bulk(p.meta + tile * 2048 + (group & 7u) * 256u, 256u);
}

// The sparse operands of a block.  A lane's 32 columns are the groups G0 .. G7; the instruction of step s (0, 1) takes
// {G[s], G[4 + s]} as its word for contraction positions 8 q .. and {G[2 + s], G[6 + s]} for 32 + 8 q .. .  On the
// activation side position 4 q' + 16 j .. is then word s + 2 (j / 2) of chunk q' (j even) or 4 + q' (j odd).
struct FewSparseOps {
    uint32_t a[2][4];                // [step][operand word]
    uint32_t e[2];                   // metadata
};
template <int WT>
__device__ __forceinline__ void few_sparse_ops(const FewBlock<WT>& b, uint32_t lane, FewSparseOps& o) {
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        if constexpr (WT == kFewSparse) {
            const uint4 w = b.w[row];
            o.a[0][row] = __byte_perm(w.x, w.z, 0x5410);
            o.a[1][row] = __byte_perm(w.x, w.z, 0x7632);
            o.a[0][row + 2] = __byte_perm(w.y, w.w, 0x5410);
            o.a[1][row + 2] = __byte_perm(w.y, w.w, 0x7632);
        } else {
            // group j = nibble j, two 2-bit values t = v + 1: spread to bytes, subtract 1 without borrows between bytes
#pragma unroll
            for (int j = 0; j < 4; ++j) {                                    // {G[j], G[4 + j]}
                const uint32_t t = (((b.w[row] >> (4 * j)) & 0x000F000Fu) * 65u) & 0x03030303u;
                o.a[j & 1][row + 2 * (j >> 1)] = (t + 0x7F7F7F7Fu) ^ 0x80808080u;
            }
        }
    }
    // Metadata of row g + 8 (lane & 1), contraction positions 32 h .. 32 h + 31 with h = (lane >> 1) & 1: nibble s of bytes
    // 4 q + 2 e + h of the row's 16, in the order (q, e).
    const uint4 m = b.m;
    const uint32_t sel = (lane & 2u) ? 0x7531u : 0x6420u;
    const uint32_t t0 = __byte_perm(m.x, m.y, sel), t1 = __byte_perm(m.z, m.w, sel);
    constexpr uint32_t kLow = 0x000F000Fu;                                   // bytes 0 and 2 of the words below matter
    auto pick = [](uint32_t a, uint32_t b2) { return (a & kLow) | (b2 & ~kLow); };
    o.e[0] = __byte_perm(pick(t0, t0 >> 4), pick(t1, t1 >> 4), 0x6420);
    o.e[1] = __byte_perm(pick(t0 >> 4, t0 >> 8), pick(t1 >> 4, t1 >> 8), 0x6420);
}

// One block of weights against the activations of 8 NT tokens (bw[nt]: words of chunk q, then of chunk 4 + q).
template <int WT, int NT>
__device__ __forceinline__ void few_mma(const FewBlock<WT>& b, uint32_t lane, const uint32_t (&bw)[NT][8], int (&acc)[NT][4]) {
    if constexpr (WT == kFewDense) {
        const uint4 l0 = b.w[0][0], h0 = b.w[0][1], l1 = b.w[1][0], h1 = b.w[1][1];
        const uint32_t a0[4] = {l0.x, l0.y, l0.z, l0.w}, a1[4] = {l1.x, l1.y, l1.z, l1.w}, a2[4] = {h0.x, h0.y, h0.z, h0.w}, a3[4] = {h1.x, h1.y, h1.z, h1.w};
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) mma_m16n8k32(acc[nt], a0[s], a1[s], a2[s], a3[s], bw[nt][s], bw[nt][4 + s]);
    } else {
        FewSparseOps o;
        few_sparse_ops<WT>(b, lane, o);
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
                mma_m16n8k64_sp(acc[nt], o.a[s], bw[nt][s], bw[nt][4 + s], bw[nt][2 + s], bw[nt][6 + s], o.e[s]);
    }
}

// 16 consecutive bf16 (two vectors) -> 16 codes in four words
__device__ __forceinline__ void few_quantise(const uint4& lo, const uint4& hi, float s_x, uint32_t* out) {
    out[0] = quant_pair2(lo.x, lo.y, s_x);
    out[1] = quant_pair2(lo.z, lo.w, s_x);
    out[2] = quant_pair2(hi.x, hi.y, s_x);
    out[3] = quant_pair2(hi.z, hi.w, s_x);
}

// NT groups of 8 tokens; W warps per CTA; D blocks of weights in flight per warp; MINB CTAs per SM (the register budget); AHEAD: the
// blocks after those go to the L2 early.
template <int WT, int NT, int W, int D, int MINB, bool FUSED, bool AHEAD>
__global__ void __launch_bounds__(32 * W, MINB)
bitlinear_gemm_few_kernel(const FewParams p) {
    constexpr int kStride = 20;                                              // words between tokens of a warp's partial sums: no bank conflicts
    __shared__ int s_red[2][W][8 * NT][kStride];                             // row groups alternate
    __shared__ float s_max[FUSED ? W : 1][8 * NT];
    __shared__ float s_scale[8 * NT];
    const uint32_t lane = threadIdx.x & 31u, g = lane >> 2, q = lane & 3u;
    const int warp = threadIdx.x >> 5;
    const int n_groups = p.N >> 4;
    const int rounds = (p.k_blocks + W - 1) / W;                             // per row group; the last one may leave warps without a block
    pdl_launch_dependents();

    // A warp's work is the sequence of its blocks over all of the CTA's row groups; D of them are always on their way, the
    // first ones from before the dependency wait.
    FewFetch<WT, W> fetch(p, lane, warp, rounds);
    FewBlock<WT> blk[D];
#pragma unroll
    for (int j = 0; j < D; ++j) fetch.next(p, lane, blk[j]);
    // (FUSED: asking the L2 for the activations here too made calls of several tokens up to 12 % slower, 2560 -> 6912 at 8 tokens 5.4 / 6.0:
    // they are there as a rule, and every CTA asks.)
    if constexpr (AHEAD) few_prefetch_next<WT, W, D>(p, lane, static_cast<uint32_t>(warp), static_cast<uint32_t>(rounds));
    pdl_wait();

    bool real[NT];                                                           // this lane's tokens exist
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) real[nt] = 8 * nt + static_cast<int>(g) < p.T;
    float s_x[NT];
    if constexpr (FUSED) {
        // per-token maximum over this warp's columns, over the quad's lanes, over the warps
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            uint32_t mx = 0u;
            if (real[nt]) {
#pragma unroll 4
                for (int kb = warp; kb < p.k_blocks; kb += W) {
                    const uint4* x = p.x_bf16 + static_cast<size_t>(8 * nt + g) * (p.k_blocks * 16) + kb * 16 + 2 * q;
                    mx = absmax8_packed(__ldg(x), absmax8_packed(__ldg(x + 1), mx));
                    mx = absmax8_packed(__ldg(x + 8), absmax8_packed(__ldg(x + 9), mx));
                }
            }
            uint32_t m = max(mx >> 16, mx & 0xFFFFu);
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
            if (q == 0u) s_max[warp][8 * nt + g] = __uint_as_float(m << 16);
        }
        __syncthreads();
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            float a = s_max[0][8 * nt + g];
#pragma unroll
            for (int w = 1; w < W; ++w) a = fmaxf(a, s_max[w][8 * nt + g]);
            const float d = fmaxf(a, kEps);
            s_x[nt] = __fdiv_rn(127.0f, d);
            if (warp == 0 && q == 0u) {
                const float sc = __fdiv_rn(d, 127.0f);
                s_scale[8 * nt + g] = sc;
                if (p.a_scale_out != nullptr && blockIdx.x == 0 && real[nt]) p.a_scale_out[8 * nt + g] = sc;
            }
        }
    } else {
        if (threadIdx.x < 8 * NT) s_scale[threadIdx.x] = static_cast<int>(threadIdx.x) < p.T ? __ldg(p.a_scale + threadIdx.x) : 0.0f;
    }
    const float w_scale = __ldg(p.w_scale);

    const uint8_t* const x_lo = FUSED ? nullptr : p.xq + g * 128u + ((q ^ g) << 4);
    const uint8_t* const x_hi = FUSED ? nullptr : p.xq + g * 128u + (((4u + q) ^ g) << 4);
    auto load_acts = [&](int kb, uint32_t (&bw)[NT][8]) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            if constexpr (FUSED) {
                uint4 v[4] = {};
                if (real[nt]) {
                    const uint4* x = p.x_bf16 + static_cast<size_t>(8 * nt + g) * (p.k_blocks * 16) + kb * 16 + 2 * q;
                    v[0] = __ldg(x); v[1] = __ldg(x + 1); v[2] = __ldg(x + 8); v[3] = __ldg(x + 9);
                }
                few_quantise(v[0], v[1], s_x[nt], &bw[nt][0]);
                few_quantise(v[2], v[3], s_x[nt], &bw[nt][4]);
            } else {
                uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
                if (real[nt]) {
                    const uint32_t o = (static_cast<uint32_t>(kb) * static_cast<uint32_t>(p.tb8) + nt) * 1024u;
                    lo = __ldg(reinterpret_cast<const uint4*>(x_lo + o));
                    hi = __ldg(reinterpret_cast<const uint4*>(x_hi + o));
                }
                bw[nt][0] = lo.x; bw[nt][1] = lo.y; bw[nt][2] = lo.z; bw[nt][3] = lo.w;
                bw[nt][4] = hi.x; bw[nt][5] = hi.y; bw[nt][6] = hi.z; bw[nt][7] = hi.w;
            }
        }
    };
    // the activations of as many blocks are asked for ahead (the same ones for every row group: from L1 after the first)
    uint32_t bw[FUSED ? 1 : D][NT][8];
    int x_round = 0;
    auto load_next_acts = [&](uint32_t (&b)[NT][8]) {
        const int kb = warp + x_round * W;
        if (kb < p.k_blocks) load_acts(kb, b);
        if (++x_round == rounds) x_round = 0;
    };
    if constexpr (!FUSED) {
#pragma unroll
        for (int j = 0; j < D; ++j) load_next_acts(bw[j]);
    }
    int acc[NT][4];
    auto clear = [&] {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[nt][i] = 0;
    };
    clear();
    int group = blockIdx.x, round = 0;
    uint32_t buf = 0;
    while (group < n_groups) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            if (group < n_groups) {
                if constexpr (FUSED) load_next_acts(bw[0]);
                if (warp + round * W < p.k_blocks) few_mma<WT, NT>(blk[j], lane, bw[FUSED ? 0 : j], acc);
                fetch.next(p, lane, blk[j]);
                if constexpr (!FUSED) load_next_acts(bw[j]);
                if (++round == rounds) {
                    // partial sums of the warps -> outputs (accumulator lane layout: features g and g + 8, tokens 2 q and
                    // 2 q + 1).  With two buffers one barrier per row group is enough: a warp comes back to a buffer only
                    // after the next group's barrier, which every warp reaches after it has read this one.
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        s_red[buf][warp][8 * nt + 2 * q][g] = acc[nt][0];
                        s_red[buf][warp][8 * nt + 2 * q + 1][g] = acc[nt][1];
                        s_red[buf][warp][8 * nt + 2 * q][g + 8] = acc[nt][2];
                        s_red[buf][warp][8 * nt + 2 * q + 1][g + 8] = acc[nt][3];
                    }
                    __syncthreads();
                    for (int o = threadIdx.x; o < 16 * p.T; o += 32 * W) {
                        const int tok = o >> 4, f = o & 15, n = group * 16 + f;
                        int sum = 0;
#pragma unroll
                        for (int w = 0; w < W; ++w) sum += s_red[buf][w][tok][f];
                        const size_t off = static_cast<size_t>(tok) * p.N + n;
                        if (p.acc_out) p.acc_out[off] = sum;
                        float v = __fmul_rn(static_cast<float>(sum), __fmul_rn(w_scale, s_scale[tok]));
                        if (p.bias) v = __fadd_rn(v, __ldg(p.bias + n));
                        if (p.out_bf16) static_cast<uint16_t*>(p.y)[off] = static_cast<uint16_t>(f32_to_bf16_rne(v));
                        else static_cast<float*>(p.y)[off] = v;
                    }
                    clear();
                    buf ^= 1u;
                    round = 0;
                    group += gridDim.x;
                }
            }
        }
    }
}

// Does the early fetch of the next blocks pay?  Not without any (groups and blocks per warp that the first D do not cover, or
// more than the next D do).  FUSED, three CTAs per SM, where the first row group's activations are still to be quantised: not while a warp
// has one block per row group (K = 640 to 1024: 1 to 5 % slower); int8-held 2:4 not beyond 1.9 groups per place (2048 -> 14336 6.5 /
// 6.7 us), nor 1.25 with K > 2048 (3072 -> 12288 8.5 / 8.8; 2560 -> 7680 6.1 / 5.9); dense, K of about 1280 to 2048, only beyond 1.3
// (2048 -> 8704 5.3 / 5.6; 2048 -> 16384 8.2 / 7.7, 2560 -> 7680 6.4 / 5.9).
template <int WT, bool FUSED, int W, int D, int MINB>
inline bool few_ahead(int k_blocks, int groups, int slots) {
    if (groups <= slots && (k_blocks <= W * D || k_blocks > 2 * W * D)) return false;
    if (!FUSED || MINB < 3) return true;
    const double per_place = static_cast<double>(groups) / slots;
    if (k_blocks <= W) return false;
    if (WT == kFewSparse) return per_place <= (k_blocks <= 2 * W ? 1.9 : 1.25);
    return k_blocks <= 10 || k_blocks > 2 * W || per_place > 1.3;
}

template <int WT, int NT, int W, int D, int MINB, bool FUSED>
inline cudaError_t launch_few_cfg(const FewParams& p, cudaStream_t stream) {
    const int groups = p.N / 16, slots = device_sm_count() * MINB;
    ++g_launch_count;
    auto kernel = bitlinear_gemm_few_kernel<WT, NT, W, D, MINB, FUSED, true>;
    // 2:4 weights always, for the sake of the order of the loads (see few_prefetch_next), which helps packed and, a little, int8-held ones
    // (2560 -> 2560 4.09 / 3.96) but not dense ones (2560 -> 3840, 8 tokens 4.75 / 4.95) nor the fused quantiser (2560 -> 3840 3.83 / 3.99).
    if constexpr (WT == kFewDense || FUSED) {
        if (!few_ahead<WT, FUSED, W, D, MINB>(p.k_blocks, groups, slots)) kernel = bitlinear_gemm_few_kernel<WT, NT, W, D, MINB, FUSED, false>;
    }
    return launch_kernel(kernel, dim3(groups < slots ? groups : slots), dim3(32 * W), 0, stream, p);
}

// Which calls run here, with what split.  All times in us for quantiser + GEMM in a decode loop (weights from HBM), this
// kernel / the cluster kernel of tcgen05 instructions at its best cluster size.
//   up to 8 tokens    all but the places at the end.  1 token: 2560 -> 2560 3.7 / 5.0, 2560 -> 6912 4.6 / 5.6, 6912 -> 2560 5.7 / 7.5,
//                     4096 -> 11008 7.8 / 8.5, 11008 -> 4096 8.4 / 10.6.
//                     With more row groups than two CTAs per SM take at once, three CTAs per SM with fewer blocks in flight
//                     each (4.6 against 5.4 for 2560 -> 6912; but 6.4 against 5.7 for 6912 -> 2560, which fits two).  Not
//                     for FUSED with K > 3072 (4096 -> 11008 10.0 against 9.5).  Dense weights of long rows already from one and a half
//                     groups per SM on (11008 -> 4096 11.5 / 10.85; 6912 -> 2560, fewer groups, 6.6 / 7.2).
//   9 to 16 tokens    only while two CTAs per SM take all row groups (4096 -> 11008 10.6 / 9.1: every CTA reads all activations,
//                     the cluster kernel's 128-row tiles read them less often).  Packed weights then always (7B MLPs, whole pass,
//                     47 / 52), int8-held ones up to 12 tokens, beyond up to K = 4352 (quantiser + GEMM,
//                     9 tokens: 3584 -> 2560 4.4 / 5.3, 6912 -> 2560 6.5 / 6.6, 11008 -> 4096 9.3 / 10.4; 12: 11008 -> 2048 8.93 / 8.97, the least gain of 28 shapes; 16:
//                     4096 -> 4096 5.6 / 6.0, but 6912 -> 2560 7.5 / 7.05; two 7B MLPs, whole pass, 44.5 / 41.8).  Dense: not
//                     (2B layers 63.5 / 59.3).  FUSED: not (6912 -> 2560 13.6 / 11.1).
//   Not where a second round of CTAs would be barely filled: it costs as much as a full one, and the clusters have none.
//                     Three CTAs per SM: int8-held 2:4 from K = 2560 on, a second round of up to a third (2560 -> 8192 6.6 / 5.7, 6912 -> 7424
//                     10.8 / 9.2; 2048 -> 8192 4.8 / 5.4), a third one likewise around K = 2560 (2560 -> 16384 8.6 / 7.5, 3072 -> 16384
//                     even); dense around K = 3072, up to a fifth (2560 -> 8704 6.9 / 6.4, 4096 -> 8704 8.7 / 9.2).  Two per SM
//                     (FUSED): long rows, up to a half (6912 -> 5120 dense, 8 tokens 15.1 / 12.1).  Packed: a second round of up to
//                     a third, K from 2560 on (8192 -> 8704 12.2 / 11.2; 2048 -> 8192 5.0 / 5.5), of up to a half, long rows (6912 ->
//                     11008 13.1 / 12.1; 4096 -> 11008 8.9 / 8.8, but 2 % slower among other matrices).
inline bool few_wide(const FewParams& p) { return p.N / 16 > 2 * device_sm_count(); }
template <int WT, bool FUSED>
inline bool few_takes(int T, int N, int K) {
    const double per_sm = static_cast<double>(N / 16) / device_sm_count();
    if (T > 8)
        return T <= 16 && !FUSED && WT != kFewDense && per_sm <= 2.0 &&
               (WT == kFewPacked || T <= 12 || K <= 4352);
    if (FUSED && K > 3072)
        return !(per_sm > 2.0 && per_sm <= (T > 4 ? 3.25 : 3.0) && (K >= 6144 || (WT == kFewDense && T > 4 && K >= 4096)));
    if (WT == kFewDense) return !(per_sm > 3.0 && per_sm <= 3.7 && K >= 2560 && K <= 3584 && (!FUSED || T > 4));
    if (WT == kFewSparse && !FUSED) return !((per_sm > 3.0 && per_sm <= 4.0 && K >= 2560) || (per_sm > 6.0 && per_sm <= 7.0 && K >= 2560 && K < 3072));
    if (WT == kFewPacked) return !((per_sm > 3.1 && per_sm <= 4.0 && K >= 2560) || (per_sm > 4.0 && per_sm <= 4.7 && K >= 6144));
    return true;
}
template <int WT, bool FUSED>
inline sbn_status launch_few(const FewParams& p, cudaStream_t stream) {
    cudaError_t err;
    if (p.T > 8) {
        if constexpr (FUSED || WT == kFewDense) return SBN_ERR_UNSUPPORTED;  // not reached: few_takes()
        else err = launch_few_cfg<WT, 2, 8, 2, 2, false>(p, stream);
    } else if ((few_wide(p) && !(FUSED && p.k_blocks > 24)) ||
               (WT == kFewDense && !FUSED && 2 * (p.N / 16) >= 3 * device_sm_count() && p.k_blocks >= 32)) {
        err = launch_few_cfg<WT, 1, 8, 2, 3, FUSED>(p, stream);
    } else {
        err = launch_few_cfg<WT, 1, 8, 4, 2, FUSED>(p, stream);
    }
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

}  // namespace sbn
