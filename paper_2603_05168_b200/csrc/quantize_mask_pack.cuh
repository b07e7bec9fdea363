// Part 1 of the path: absmean ternary quantisation (Eq. 1), 2:4 magnitude mask from the master
// weights (Eq. 2), W_eff = W_q (.) M (Eq. 3), compressed value + metadata layout.
//
// gamma needs the whole matrix before any element can be rounded, but almost every element can be
// rounded correctly from an ESTIMATE of gamma: W_q = sign(w) [ |w| >= thr(gamma) ] and only the
// few |w| that lie within a few percent of thr depend on its exact value.  One persistent kernel
// (one 768-thread CTA per SM) therefore reads W ONCE, for one matrix or a batch of them.  This file
// holds the building blocks; the kernel runs the phases as one uninterrupted stream
// (quantize_mask_pack_stream.cuh).  The phases:
//
//   sample   every CTA adds |w| over the same 256 scattered 512 B units of the matrix (128 KB,
//            L2-served for all CTAs but the first; 64 units for matrices below 33 M weights)
//            -> gamma_est, and brackets the threshold: thr_lo ~ thr(0.97 gamma_est),
//            thr_hi ~ thr(1.03 gamma_est) (0.96 / 1.04 with the small sample);
//   pass 1   every CTA owns a contiguous range of (row, 128-column) units and streams it:
//            sum|W| in fp64 (the exact gamma), top 2 of 4 per group (Eq. 2: the mask does not
//            depend on gamma), metadata, flip count, and the two kept values ternarised
//            PROVISIONALLY: |w| >= thr_hi -> +-1 and |w| < thr_lo -> 0 are final whatever gamma
//            turns out to be inside the bracket; the others (~2 % for Gaussian weights) are
//            appended as {byte position, w} to a list in shared memory;
//   exchange every CTA publishes {tag, partial sum} in the workspace and waits (bounded) until all
//            slots carry this execution's tag -- no atomics, nothing to initialise; every CTA then
//            adds the 148 partials in the same fixed order, so all get the same bits, run after
//            run.  The tag joins the host's per-call nonce with a generation word that lives in
//            the workspace and that CTA 0 advances at the end of every execution: stale slots of
//            earlier calls never match, and neither do those of an earlier REPLAY of the same
//            captured launch (whose nonce is frozen in the graph);
//   fix-up   with the exact thr: if thr_lo <= thr <= thr_hi (and the list did not overflow) only
//            the listed bytes are rewritten -- the result is exactly Eq. 1, not an approximation.
//            Otherwise (a sample that misrepresents the matrix, the 1e-5 clamp, a request for the
//            dense W_q, which needs all four weights of a group) the CTA reads its range again
//            and ternarises everything with the exact thr: slower, same result.
//
// HBM traffic per parameter: 4 B read + 0.625 B written.  16 B loads per lane, a warp covers one
// 512 B unit; a warp store covers whole 64 B (vals), 128 B (dense W_q) or 16 B (metadata) rows of
// an operand tile (tiled layouts, see layouts.cuh).
//
// Ternarisation without a per-element division: W_q = sign(w) * [ fl(|w| / scale) > 0.5 ]
// (round-half-even sends exactly 0.5 to 0, everything above to >= 1, the clamp caps at 1).
// Correctly rounded division is monotone in |w|, so there is one fp32 threshold thr with
// fl(a / scale) > 0.5  <=>  a >= thr.  thr is found once per matrix with real IEEE divisions
// and the per-element work is a compare.
#pragma once

#include <algorithm>

#include "sbn_common.cuh"
#include "layouts.cuh"

namespace sbn {

constexpr int kQmpThreads = 768;
constexpr int kQmpWarps = kQmpThreads / 32;
constexpr int kQmpMaxCtas = kNumSMs;                       // one CTA per SM, all co-resident
constexpr int kQmpSampleUnits = 256;                       // units in the gamma_est sample of a large matrix
constexpr float kQmpBracket = 0.03f;                       // gamma_est * (1 -+ this) brackets gamma
// Matrices below 2^18 units (33.5 M weights) are sampled at a quarter of that with a wider bracket:
// there the sample is a visible part of the kernel's time (2.5 us of ~25), and 8192 weights still put
// the bracket at 4.8 standard errors of the mean for Gaussian weights.  Large matrices keep the
// larger sample, which also holds for heavy-tailed weights.
constexpr int kQmpSampleUnitsSmall = 64;
constexpr float kQmpBracketSmall = 0.04f;
constexpr uint32_t kQmpSmallMatrixUnits = 1u << 18;
__host__ __device__ inline uint32_t qmp_sample_units(uint32_t num_units) {
    const uint32_t want = num_units < kQmpSmallMatrixUnits ? kQmpSampleUnitsSmall : kQmpSampleUnits;
    return num_units < want ? num_units : want;
}

struct __align__(16) QmpSlot {   // one per CTA, 16 B: the stream kernel writes and reads it as one 128-bit word
    unsigned long long nonce;    // tag of the execution that wrote `partial`
    double partial;              // this CTA's sum |W|
};
// What a single-matrix call leaves behind for the next call on the same workspace: the scale it found,
// tagged with the matrix it belongs to.  The next call on the same matrix (a training loop re-packs the
// same buffers every step) takes it as its estimate of gamma -- no sample, a narrow bracket -- exactly as
// if the caller had passed it as a hint; anything else in these bytes (an uninitialised workspace, another
// matrix) fails the tag and is ignored.
struct __align__(16) QmpMemo {
    unsigned long long magic;
    const void* W;
    uint32_t num_units;
    float scale;
};
constexpr unsigned long long kQmpMemoMagic = 0x71A93C5E2D84B6F1ull;
struct QmpWorkspace {            // layout of the caller's workspace
    QmpSlot slot[kQmpMaxCtas];
    unsigned long long generation;   // advanced by one per execution on this workspace (any start value)
    unsigned long long pad_;
    QmpMemo memo;
    unsigned long long pad2_;
};
// Tag of one execution: the call's nonce (low word, never 0) under the workspace's generation.
__device__ __forceinline__ unsigned long long qmp_tag(unsigned long long nonce, unsigned long long generation) {
    return (generation << 32) | (nonce & 0xFFFFFFFFull);
}

__device__ __forceinline__ unsigned long long global_timer_ns_qmp() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Eq. 2 for one group: the two largest |w| of four (ranking on the fp32 master weights; on equal
// magnitudes the lower column wins).  Returns the nibble i0 | i1 << 2 (i0 < i1) and the two kept
// weights in column order.  The winners of the pairs (0,1) and (2,3) are the answer unless the
// loser of one pair still beats the winner of the other:
//   min(a0,a1) >= max(a2,a3)  ->  columns 0,1   (a tie goes to the lower column, hence >=)
//   min(a2,a3) >  max(a0,a1)  ->  columns 2,3   (and hence > here)
__device__ __forceinline__ uint32_t select_pair(const float4 w, float& v0, float& v1) {
    const float a0 = fabsf(w.x), a1 = fabsf(w.y), a2 = fabsf(w.z), a3 = fabsf(w.w);
    const bool both01 = fminf(a0, a1) >= fmaxf(a2, a3);
    const bool both23 = fminf(a2, a3) > fmaxf(a0, a1);
    const bool first0 = a0 >= a1 || both01;
    const bool second2 = a2 >= a3 && !both23;
    v0 = both23 ? w.z : (first0 ? w.x : w.y);
    v1 = both01 ? w.y : (second2 ? w.z : w.w);
    return (both23 ? 2u : (first0 ? 0u : 1u)) | (both01 ? 4u : (second2 ? 8u : 12u));
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// 0xFF where the word is negative, a byte per word (byte permutes in sign-replication mode).
__device__ __forceinline__ uint32_t sign_bytes4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return prmt(prmt(a, b, 0x00FBu), prmt(c, d, 0x00FBu), 0x5410u);
}
__device__ __forceinline__ uint32_t sign_bytes4(float a, float b, float c, float d) {
    return sign_bytes4(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c), __float_as_uint(d));
}
// Eight byte masks -> eight bits.
__device__ __forceinline__ uint32_t qmp_byte_bits(uint32_t lo, uint32_t hi) {
    return (((lo & 0x08040201u) | (hi & 0x80402010u)) * 0x01010101u) >> 24;
}
// Two bf16 in a word: magnitudes, sign bits, the permute that turns the four sign bits of two words into four byte masks (low half
// of the first word first).
constexpr uint32_t kAbs2 = 0x7FFF7FFFu, kGuard2 = 0x80008000u, kSign2 = 0xFDB9u;
// |a| - |b| for two bf16 at once: only the sign bits (15 and 31) are used -- rounding cannot change them, and equal magnitudes
// give +0.  It runs on the FMA pipe, where nothing else waits: pass 1 is bound by the ALU pipe.
__device__ __forceinline__ uint32_t sub_abs_bf16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("{\n\t.reg .b32 x, y;\n\tabs.bf16x2 x, %1;\n\tabs.bf16x2 y, %2;\n\tsub.rn.bf16x2 %0, x, y;\n\t}" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Three-input minima (one instruction each on this architecture).
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint32_t umin8(const uint32_t (&e)[8]) {
    return __vimin3_u32(__vimin3_u32(e[0], e[1], e[2]), __vimin3_u32(e[3], e[4], e[5]), min(e[6], e[7]));
}

// Eq. 1 for four elements as four bytes (+1 -> 0x01, -1 -> 0xFF, 0 -> 0x00; thr: see the header),
// lowest byte = first argument.  The sign bytes come from byte permutes in sign-replication mode.
__device__ __forceinline__ uint32_t ternary_bytes4(float w0, float w1, float w2, float w3, float thr) {
    const uint32_t s01 = prmt(__float_as_uint(w0), __float_as_uint(w1), 0x00FBu);   // bytes 0,1: 0xFF if negative
    const uint32_t s23 = prmt(__float_as_uint(w2), __float_as_uint(w3), 0x00FBu);
    const uint32_t sgn = prmt(s01, s23, 0x5410u);
    const uint32_t keep = (fabsf(w0) >= thr ? 0x000000FFu : 0u) | (fabsf(w1) >= thr ? 0x0000FF00u : 0u) |
                          (fabsf(w2) >= thr ? 0x00FF0000u : 0u) | (fabsf(w3) >= thr ? 0xFF000000u : 0u);
    return (sgn | 0x01010101u) & keep;
}
__device__ __forceinline__ uint32_t ternary_bytes2(float w0, float w1, float thr) {
    const uint32_t sgn = prmt(__float_as_uint(w0), __float_as_uint(w1), 0x00FBu);
    const uint32_t keep = (fabsf(w0) >= thr ? 0x00FFu : 0u) | (fabsf(w1) >= thr ? 0xFF00u : 0u);
    return (sgn | 0x0101u) & keep;
}

__device__ __forceinline__ uint32_t nibble_to_mask(uint32_t nib) {
    return (1u << (nib & 3u)) | (1u << ((nib >> 2) & 3u));
}

__device__ __forceinline__ double abs_sum4(const float4 v) {
    return ((double)fabsf(v.x) + (double)fabsf(v.y)) + ((double)fabsf(v.z) + (double)fabsf(v.w));
}

// One matrix of a batch (device-visible copy of the call's arguments).
struct QmpDesc {
    const void* W;                     // fp32 [N][K], or bf16 [N][K] when w_bf16
    uint16_t* vals;
    uint8_t* meta;
    float* w_scale;
    uint32_t* dense_q;                 // or null
    const uint8_t* prev_meta;          // or null
    unsigned long long* flip_bits;     // or null
    const float* gamma_hint;           // or null: the caller's estimate of gamma (e.g. the previous step's scale)
    uint32_t num_units;                // N * K / 128
    uint32_t KB;                       // K / 128
    uint32_t w_bf16;                   // master weights are bf16 (Sec. 2.2 keeps them "e.g. in bf16")
    uint32_t kb_magic;                 // qmp_magic(KB)
};
// Division by a number the host knows: a 32-bit division is 25 dependent instructions, and one thread's chain of them
// is what a short call waits for at its start.
__host__ __device__ inline uint32_t qmp_magic(uint32_t d) { return d > 1u ? 0xFFFFFFFFu / d + 1u : 0u; }
// x / d and its remainder: magic / 2^32 lies above 1 / d by less than 2^-32, so the estimate is at most one too large.
__device__ __forceinline__ uint32_t qmp_div(uint32_t x, uint32_t d, uint32_t magic, uint32_t& rem) {
    uint32_t q = magic != 0u ? __umulhi(x, magic) : x;
    rem = x - q * d;
    if (rem >= d) { --q; rem += d; }
    return q;
}

struct QmpRange {                      // this CTA's share of one matrix
    uint32_t u_begin, u_end;
};
struct QmpEntry {                      // one undecided kept value
    uint32_t byte_off;                 // its byte in vals
    float w;
};

// One group (4 consecutive weights) of unit u for lane `lane` (a warp covers the unit's 32 groups).
template <bool BF16>
__device__ __forceinline__ float4 qmp_load_group(const void* W, size_t u, int lane) {
    if constexpr (BF16) {
        const uint2 v = __ldg(static_cast<const uint2*>(W) + u * 32 + lane);
        return make_float4(bf16lo_to_f32(v.x), bf16hi_to_f32(v.x), bf16lo_to_f32(v.y), bf16hi_to_f32(v.y));
    } else {
        return __ldg(static_cast<const float4*>(W) + u * 32 + lane);
    }
}
// Two adjacent groups of unit u for lane l16 of a half-warp (16 lanes cover the unit).
template <bool BF16>
__device__ __forceinline__ void qmp_load_group_pair(const void* W, size_t u, uint32_t l16, float4& a, float4& b) {
    if constexpr (BF16) {
        const uint4 v = __ldg(static_cast<const uint4*>(W) + u * 16 + l16);
        a = make_float4(bf16lo_to_f32(v.x), bf16hi_to_f32(v.x), bf16lo_to_f32(v.y), bf16hi_to_f32(v.y));
        b = make_float4(bf16lo_to_f32(v.z), bf16hi_to_f32(v.z), bf16lo_to_f32(v.w), bf16hi_to_f32(v.w));
    } else {
        const float4* src = static_cast<const float4*>(W) + u * 32 + 2 * l16;
        a = __ldg(src);
        b = __ldg(src + 1);
    }
}

__device__ __forceinline__ QmpRange qmp_range(const QmpDesc& d, uint32_t grid_magic) {
    QmpRange r;
    uint32_t rem;
    const uint32_t per = qmp_div(d.num_units + gridDim.x - 1u, gridDim.x, grid_magic, rem);
    r.u_begin = min(d.num_units, blockIdx.x * per);
    r.u_end = min(d.num_units, r.u_begin + per);
    return r;
}

// Ternarise a whole range again with the exact threshold (the path taken when the bracket missed,
// the list overflowed or the dense W_q is wanted): a warp per unit, four units at a time, newest
// first (what pass 1 read last is still in L2).
template <bool BF16>
__device__ __forceinline__ void qmp_pass2_full(const QmpDesc& d, const QmpRange rg, float thr) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const uint32_t KB = d.KB;
    const uint32_t n_units = rg.u_end - rg.u_begin;
    const bool write_dense = d.dense_q != nullptr;
    const int step_n = static_cast<int>(kQmpWarps / KB), step_kb = static_cast<int>(kQmpWarps % KB);
    int n_cur = 0, kb_cur = 0;
    if (static_cast<uint32_t>(warp) < n_units) {
        const uint32_t u_first = rg.u_begin + (n_units - 1 - warp);
        n_cur = static_cast<int>(u_first / KB);
        kb_cur = static_cast<int>(u_first - static_cast<uint32_t>(n_cur) * KB);
    }
    for (uint32_t i0 = warp; i0 < n_units; i0 += 4 * kQmpWarps) {
        float4 w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t i = i0 + q * kQmpWarps;
            w[q] = (i < n_units) ? qmp_load_group<BF16>(d.W, rg.u_begin + (n_units - 1 - i), lane)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t i = i0 + q * kQmpWarps;
            if (i < n_units) {
                const size_t tile_idx = static_cast<size_t>(static_cast<uint32_t>(n_cur) >> 7) * KB + static_cast<uint32_t>(kb_cur);
                const uint32_t rr = static_cast<uint32_t>(n_cur) & 127u;
                n_cur -= step_n;
                kb_cur -= step_kb;
                if (kb_cur < 0) { kb_cur += static_cast<int>(KB); --n_cur; }
                float k0, k1;
                select_pair(w[q], k0, k1);
                // compressed columns 2*lane, 2*lane+1 of this 64 B tile row
                d.vals[((tile_idx << 13) + vals_in_tile(rr, 2u * lane)) >> 1] = static_cast<uint16_t>(ternary_bytes2(k0, k1, thr));
                if (write_dense)
                    d.dense_q[((tile_idx << 14) + sw128_in_tile(rr, 4u * lane)) >> 2] =
                        ternary_bytes4(w[q].x, w[q].y, w[q].z, w[q].w, thr);
            }
        }
    }
}

// Copies up to kQmpDescChunk job descriptors, passed by value, into the batch workspace: the batched
// call hands its jobs to the device without a host-side staging copy.
constexpr int kQmpDescChunk = 48;
struct QmpDescChunk {
    QmpDesc d[kQmpDescChunk];
};
static_assert(sizeof(QmpDescChunk) <= 4000, "descriptor chunk must fit the kernel parameter space");
__global__ void __launch_bounds__(64)
qmp_store_descs_kernel(const QmpDescChunk chunk, QmpDesc* __restrict__ dst, int n) {
    pdl_wait();                        // the previous user of the workspace has finished; no early start for successors
    if (threadIdx.x < static_cast<unsigned>(n)) dst[threadIdx.x] = chunk.d[threadIdx.x];
}

// Per-call nonce: unique within the process, low 32 bits never 0.
inline unsigned long long qmp_next_nonce() {
    static std::atomic<unsigned long long> counter{0x5B4E0000ull};
    unsigned long long n = counter.fetch_add(1) + 1;
    if ((n & 0xFFFFFFFFull) == 0ull) n = counter.fetch_add(1) + 1;
    return n;
}

inline QmpDesc qmp_make_desc(const void* W, bool w_bf16, int N, int K, int8_t* vals, uint8_t* meta, float* w_scale,
                             int8_t* dense_q, const uint8_t* prev_meta, unsigned long long* flip_bits,
                             const float* gamma_hint = nullptr) {
    QmpDesc d;
    d.gamma_hint = gamma_hint;
    d.W = W;
    d.w_bf16 = w_bf16 ? 1u : 0u;
    d.vals = reinterpret_cast<uint16_t*>(vals);
    d.meta = meta;
    d.w_scale = w_scale;
    d.dense_q = reinterpret_cast<uint32_t*>(dense_q);
    d.prev_meta = prev_meta;
    d.flip_bits = prev_meta ? flip_bits : nullptr;
    d.num_units = static_cast<uint32_t>(static_cast<size_t>(N) * K / 128);
    d.KB = static_cast<uint32_t>(K / 128);
    d.kb_magic = qmp_magic(d.KB);
    return d;
}

}  // namespace sbn
