// Part 1 (Eq. 1-3) for one matrix or a batch, as ONE uninterrupted stream over the weights; 2:4 and 6:8 patterns.
//
// quantize_mask_pack.cuh explains the single-read scheme (bracketed threshold, provisional values,
// fix-up list, exact fallback).  What costs time beside the stream itself is latency: the sample that
// brackets the threshold (a round trip to HBM), the exchange of the per-CTA partial sums (two more),
// the fix-up of the listed values, and a handful of CTA-wide barriers per matrix -- 5 to 7 us per
// matrix, a third of a batch of 2B-shaped matrices and more for small ones.  Here none of that stops
// the stream:
//
//   warp 20       the loader: one lane copies the CTA's range of matrix 0, 1, 2, ... into a ring of shared-
//                 memory stages (20 KB = 40 units of fp32 or 80 of bf16 weights each, six stages) with bulk
//                 copies that count their bytes on a stage's `full` barrier; it refills a stage as soon as the
//                 warps that use it have released it (`empty` barrier).  The loads cost no registers and no
//                 issue slots, and run ahead across matrices.
//   warps 0..19   pass 1 of matrix 0, 1, 2, ... back to back: two teams of 10 warps take the stages in turn
//                 (fixed order of additions: the partial sums are reproducible bit for bit); no CTA-wide barrier
//                 between matrices.  A warp leaves its sum |W| and flip count of matrix m in shared memory and
//                 arrives on the list slot's `done` barrier.  (Seven teams of four warps were tried, to keep more
//                 warps busy while some are between two matrices: their 8 KB copies stream fp32 weights at
//                 3.3 TB/s, 20 KB ones and longer at 4.7.)
//   warp 21       the finisher.  For matrix m, in this order:
//                   wait until the 20 computing warps have arrived for m, add their sums in a fixed
//                   order, publish {tag, partial} in the workspace;
//                   exchange of matrix m - 1 (published by every CTA one matrix ago, so the slots are
//                   there already), exact gamma, scale, threshold; fix-up of the listed values of
//                   m - 1, or a note that m - 1 needs the exact second pass; its list becomes free.
//                 All of it runs under pass 1 of the following matrices.
//   warps 22, 23  the scouts take turns to prepare the matrices ahead: descriptor, what the computing warps need
//                 to know (`job`), bracket from the caller's hint or from a sample of the matrix.  Up to seven
//                 matrices ahead, so neither is ever waited for.  When the finisher did this too it took 7 us per
//                 matrix, and small matrices (1 us of streaming) waited for it.
//   three lists   matrix m - 1 is being fixed up while m waits and m + 1 is being written; a computing
//                 warp starts matrix m only once m - 3 is fixed (its list slot is free) and the job
//                 of m exists -- both normally long done.
//   first look    a single long matrix without a hint: the finishers exchange what the first stages of all CTAs said about
//                 the mean, while pass 1 runs, and narrow the bracket (qmp_look_report).
//   tail          after the last matrix every warp joins: fix-up of the last matrix, then
//                 the exact second passes that were put off (bracket missed, list overflow, or the
//                 dense W_q wanted), all threads working.
//
// Every wait is bounded; one that runs out raises the CTA's abort flag and the device status word.
#pragma once

#include "quantize_mask_pack.cuh"
#include "quantize_mask_pack68.cuh"

namespace sbn {

// 20 compute, then the loader, the finisher and two scouts.  More warps (28, until the registers are used up at 64 per thread)
// make this slower: pass 1 is bound by its instructions, and with 80 registers it has fewer of them.  28 warps and four stages
// / 20 and six, us: one matrix 2560 -> 2560 fp32 15.7 / 14.9, bf16 14.7 / 13.6, 4096 -> 11008 bf16 39.8 / 39.0; 14 tensors with hints
// fp32 133.7 / 130.3, bf16 122.1 / 114.4, without 156 / 147 and 152 / 141.  24 and 16 warps lie between.
constexpr int kQmpStreamWarps = 20;
constexpr int kQmpLoaderWarp = kQmpStreamWarps;
constexpr int kQmpFinisherWarp = kQmpStreamWarps + 1;
constexpr int kQmpScoutWarp = kQmpStreamWarps + 2;
constexpr int kQmpScouts = kQmpWarps - kQmpScoutWarp;
constexpr int kQmpLists = 3;
constexpr int kQmpWarpListCap = 196;                       // undecided entries per computing warp and matrix, three lists in use
constexpr int kQmpListEntries = kQmpStreamWarps * kQmpWarpListCap;
// A launch of one or two matrices uses one or two of the three lists, each that much larger.
__host__ __device__ inline uint32_t qmp_list_cap(int count) {
    return static_cast<uint32_t>(count >= kQmpLists ? kQmpWarpListCap : kQmpLists * kQmpWarpListCap / count);
}
constexpr int kQmpTeams = 2;
constexpr int kQmpTeamWarps = kQmpStreamWarps / kQmpTeams;
static_assert(kQmpTeams * kQmpTeamWarps == kQmpStreamWarps && kQmpScouts >= 1, "who does what");
constexpr int kQmpStepUnits = 4 * kQmpTeamWarps;           // one unit per quarter-warp: what a team takes in one step
// Whole turns of the teams: a slot always belongs to the same team.  A team that comes to a slot's next use has then
// itself seen the use before land, so the parity of the slot's barrier says which use it is.  (With slots that
// wander from team to team a use could be taken for landed while the one before, another team's, was still on its way.)
constexpr int kQmpStages = 3 * kQmpTeams;
constexpr int kQmpStageBytes = kQmpStepUnits * 512;        // one step of fp32 units, or two of bf16 units
constexpr int kQmpStreamSmemBytes = kQmpStages * kQmpStageBytes + kQmpLists * kQmpListEntries * 8;
constexpr int kQmpMaxBatch = 512;                          // thresholds of put-off second passes live in shared memory
constexpr int kQmpJobs = 8;                                // matrices m - 1 .. m + 6 have a job on chip

// What the computing warps need to know about a matrix, in shared memory (a field of the kernel parameters or
// of a descriptor in global memory is a miss of its own, and all of a CTA's warps would wait for it).
struct QmpJob {
    unsigned char* vals;
    uint8_t* meta;
    const uint8_t* prev;                                   // or null
    uint32_t KB;
    uint32_t kb_magic;                                     // qmp_magic(KB)
    uint32_t units;                                        // of this CTA's range
    uint32_t n0, kb0;                                      // row and 128-column block of its first unit
    uint32_t rep_n, rep_kb;                                // kQmpStepUnits units further (next step of a stage)
    uint32_t next_n, next_kb;                              // from the last step of a stage to the first of the team's next one
    uint32_t bf16;
    float2 bracket;                                        // around the threshold: lo, hi; may become narrower under way (one 8-byte store)
    int ready;                                             // m + 1 once the rest is that of matrix m
};

struct QmpStreamShared {
    double warp_sum[kQmpLists][kQmpStreamWarps][8];
    unsigned int warp_flips[kQmpLists][kQmpStreamWarps];
    unsigned int warp_listed[kQmpLists][kQmpStreamWarps];  // entries of each warp's list (may exceed its capacity)
    QmpJob job[kQmpJobs];
    int fixed_upto;                                        // matrices < fixed_upto are finished: their list slot is free
    int abort;
    float thr_tail;
    int tail_second_pass;
    float sample[kQmpWarps];
    float look_sum[kQmpStreamWarps];                       // sum |w| of each warp's first step of matrix 0
    int look;                                              // the first look is wanted (matrix 0 has no hint)
    unsigned long long bar_look;
    unsigned long long bar_full[kQmpStages];               // a stage's bytes have landed
    unsigned long long bar_empty[kQmpStages];              // the team's warps are done with a stage
    unsigned long long bar_done[kQmpLists];                // the computing warps are done with the matrix in this slot
    uint32_t ring_issued, ring_used;                       // the loader's copies of this launch, and its ring position
    float thr_second_pass[kQmpMaxBatch];                   // >= 0: this matrix needs the exact second pass with this threshold
};
static_assert(kQmpStreamSmemBytes + sizeof(QmpStreamShared) + 256 * sizeof(uint2) <= 232448, "shared memory overflow");

// mbarrier and bulk-copy wrappers of the stage ring
__device__ __forceinline__ uint32_t qmp_smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void qmp_mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void qmp_mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void qmp_mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool qmp_mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for a barrier phase; gives up (false) when the CTA aborts or the limit runs out.  With
// `drain` it ignores the abort flag: the loader uses it to see its last copies land before the CTA leaves.
__device__ __forceinline__ bool qmp_mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, bool drain = false) {
    if (qmp_mbar_try_wait(bar, parity)) return true;
    unsigned long long t0 = 0ull;
    unsigned int spins = 0;
    while (!qmp_mbar_try_wait(bar, parity)) {
        if ((++spins & 0x3FFu) == 0u) {
            if (!drain && *abort_flag) return false;
            const unsigned long long now = global_timer_ns_qmp();
            if (t0 == 0ull) {
                t0 = now;
            } else if (now - t0 > *reinterpret_cast<volatile unsigned long long*>(&g_wait_limit_ns)) {
                *abort_flag = 1;
                atomicExch(&g_device_status, static_cast<int>(SBN_ERR_TIMEOUT));
                return false;
            }
        }
    }
    return true;
}
__device__ __forceinline__ float4 qmp_lds128(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
// The loader's position in the ring: the number of stages used so far gives the slot and the parity of its current use.
struct QmpRing {
    uint32_t used;
    __device__ __forceinline__ uint32_t stage() const { return used % kQmpStages; }
    __device__ __forceinline__ uint32_t phase() const { return (used / kQmpStages) & 1u; }
    __device__ __forceinline__ void advance() { ++used; }
};

// Matrix m of the batch: the first kQmpInlineDescs travel with the launch (kernel parameters: a batch
// that small needs no kernel that stores its descriptors first), `rest` holds 1, 2, ... in global memory.
constexpr int kQmpInlineDescs = 8;
struct QmpInlineDescs {
    QmpDesc d[kQmpInlineDescs];
};
struct QmpBatch {
    const QmpInlineDescs& inl;
    const QmpDesc* rest;
};
__device__ __forceinline__ QmpDesc qmp_desc_of(const QmpBatch& b, int m) {
    return m < kQmpInlineDescs ? b.inl.d[m] : b.rest[m - 1];
}

// Bounded wait for a shared-memory word (written by another warp of this CTA) to reach `want`.
__device__ __forceinline__ bool qmp_wait_ge(volatile int* word, int want, volatile int* abort_flag) {
    if (*word >= want) return true;
    unsigned long long t0 = 0ull;
    unsigned int spins = 0;
    while (*word < want) {
        __nanosleep(64);
        if ((++spins & 0x3Fu) == 0u) {
            if (*abort_flag) return false;
            const unsigned long long now = global_timer_ns_qmp();
            if (t0 == 0ull) {
                t0 = now;
            } else if (now - t0 > *reinterpret_cast<volatile unsigned long long*>(&g_wait_limit_ns)) {
                *abort_flag = 1;
                atomicExch(&g_device_status, static_cast<int>(SBN_ERR_TIMEOUT));
                return false;
            }
        }
    }
    return true;
}

// lo / hi of the bracket around the threshold that gamma_est predicts (see quantize_mask_pack.cuh).  An
// estimate from the caller (the scale of the previous training step, Sec. 2.2: the weights move by a
// learning-rate-sized step) gets a bracket six times narrower than one from a sample: almost no warp then
// meets an undecided value, and listing them is a tenth of pass 1's instructions otherwise.  A hint that
// is off by more than that costs the exact second pass, never the result.
constexpr float kQmpBracketHint = 0.005f;
__device__ __forceinline__ float2 qmp_bracket(float gamma_est, float b) {
    return make_float2(0.5f * fmaxf(gamma_est * (1.0f - b), kEps) * (1.0f - 1e-6f), 0.5f * fmaxf(gamma_est * (1.0f + b), kEps) * (1.0f + 1e-6f));
}
__device__ __forceinline__ float2 qmp_bracket_from(float gamma_est, uint32_t num_units, bool from_hint, bool wide = false) {
    return qmp_bracket(gamma_est, from_hint ? kQmpBracketHint : ((wide || num_units < kQmpSmallMatrixUnits) ? kQmpBracketSmall : kQmpBracket));
}

// The caller's estimate of gamma, if it gave a usable one.
__device__ __forceinline__ bool qmp_hint_usable(float g) { return g > 0.0f && g < 3.0e38f; }
__device__ __forceinline__ bool qmp_hint(const QmpDesc& d, float& g) {
    if (d.gamma_hint == nullptr) return false;
    g = *reinterpret_cast<const volatile float*>(d.gamma_hint);
    return qmp_hint_usable(g);
}

// gamma_est of the first matrix: mean |w| over qmp_sample_units units scattered over it (the same units in every
// CTA; a multiplicative hash keeps them off any row / column-block period).  In two halves, so that something can
// be started between asking for the sample and using it: all of a thread's sample loads are issued (into v), later
// they are added up over the CTA -- one barrier, after which every warp adds the partial sums of all warps itself.
// The values stay as loaded (bf16: two words) until they are added up: a conversion next to the load makes every
// load of a thread wait for the one before (64 trips in a row, 60 us, for a warp's sample of a bf16 matrix).
__device__ __forceinline__ float4 qmp_load_group_raw(const QmpDesc& d, uint32_t u, int lane) {
    if (d.w_bf16 == 0u) return __ldg(static_cast<const float4*>(d.W) + static_cast<size_t>(u) * 32 + lane);
    const float2 v = __ldg(static_cast<const float2*>(d.W) + static_cast<size_t>(u) * 32 + lane);
    return make_float4(v.x, v.y, 0.0f, 0.0f);
}
__device__ __forceinline__ float qmp_abs_sum_raw(const bool bf16, const float4 v) {
    if (!bf16) return (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
    const uint32_t a = __float_as_uint(v.x), b = __float_as_uint(v.y);
    return (fabsf(bf16lo_to_f32(a)) + fabsf(bf16hi_to_f32(a))) + (fabsf(bf16lo_to_f32(b)) + fabsf(bf16hi_to_f32(b)));
}
// Where the sampled units lie: number s in [s stride, (s + 1) stride).
struct QmpSamplePlaces {
    uint32_t n_s, stride;
    float inv;
    __device__ __forceinline__ explicit QmpSamplePlaces(uint32_t num_units) : n_s(qmp_sample_units(num_units)) {
        // the usual counts are powers of two, a matrix of fewer units is read whole
        stride = n_s == kQmpSampleUnits ? num_units / kQmpSampleUnits : (n_s == kQmpSampleUnitsSmall ? num_units / kQmpSampleUnitsSmall : 1u);
        inv = __frcp_rn(static_cast<float>(stride));
    }
    __device__ __forceinline__ uint32_t unit(uint32_t s) const {
        const uint32_t h = (s * 2654435761u) >> 8;                                       // h mod stride; h < 2^24: the quotient is one off at most
        int rem = static_cast<int>(h - __float2uint_rz(static_cast<float>(h) * inv) * stride);
        if (rem < 0) rem += static_cast<int>(stride);
        if (rem >= static_cast<int>(stride)) rem -= static_cast<int>(stride);
        return s * stride + static_cast<uint32_t>(rem);
    }
};
// The loads carry no condition and no conversion (see above): a place beyond the sample is read as its last unit and left out
// of the sum.  Small samples take three of a thread's loads, large ones all eleven.
constexpr int kQmpSamplePerWarp = (kQmpSampleUnits + kQmpWarps - 1) / kQmpWarps, kQmpSamplePerWarpSmall = (kQmpSampleUnitsSmall + kQmpWarps - 1) / kQmpWarps;
template <int FIRST, int LAST>
__device__ __forceinline__ void qmp_sample_loads(const QmpDesc& d, const QmpSamplePlaces& places, float4 (&v)[kQmpSamplePerWarp]) {
    const int lane = threadIdx.x & 31;
    const uint32_t warp = threadIdx.x >> 5;
    uint32_t u[LAST - FIRST];
#pragma unroll
    for (int i = FIRST; i < LAST; ++i) u[i - FIRST] = places.unit(min(warp + i * kQmpWarps, places.n_s - 1u));
    if (d.w_bf16 != 0u) {
#pragma unroll
        for (int i = FIRST; i < LAST; ++i)
            asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v[i].x), "=f"(v[i].y) : "l"(static_cast<const float2*>(d.W) + static_cast<size_t>(u[i - FIRST]) * 32 + lane));
    } else {
#pragma unroll
        for (int i = FIRST; i < LAST; ++i)
            asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[i].x), "=f"(v[i].y), "=f"(v[i].z), "=f"(v[i].w) : "l"(static_cast<const float4*>(d.W) + static_cast<size_t>(u[i - FIRST]) * 32 + lane));
    }
}
__device__ __forceinline__ void qmp_sample_issue(const QmpDesc& d, float4 (&v)[kQmpSamplePerWarp]) {
    const QmpSamplePlaces places(d.num_units);
    qmp_sample_loads<0, kQmpSamplePerWarpSmall>(d, places, v);
    if (places.n_s > kQmpSampleUnitsSmall) qmp_sample_loads<kQmpSamplePerWarpSmall, kQmpSamplePerWarp>(d, places, v);
}
__device__ __forceinline__ float qmp_sample_finish(const QmpDesc& d, const float4 (&v)[kQmpSamplePerWarp], float* s_sample) {
    const uint32_t n_s = qmp_sample_units(d.num_units), warp = threadIdx.x >> 5;
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < kQmpSamplePerWarp; ++i)
        if (warp + i * kQmpWarps < n_s) acc += qmp_abs_sum_raw(d.w_bf16 != 0u, v[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) s_sample[threadIdx.x >> 5] = acc;
    __syncthreads();
    float t = (threadIdx.x & 31) < kQmpWarps ? s_sample[threadIdx.x & 31] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    return t / (static_cast<float>(n_s) * 128.0f);
}

// gamma_est by ONE warp (a scout, for matrices 1, 2, ... of a batch without hints) from the first
// kQmpSampleUnitsSmall of qmp_sample_issue's scattered units, eight in flight at a time.  The smaller sample gets the
// wider bracket (qmp_bracket_from, `wide`).
__device__ __forceinline__ float qmp_sample_gamma_warp(const QmpDesc& d, int lane) {
    const QmpSamplePlaces places(d.num_units);
    const uint32_t n_s = min(places.n_s, static_cast<uint32_t>(kQmpSampleUnitsSmall));
    float acc = 0.0f;
#pragma unroll 1
    for (uint32_t s0 = 0; s0 < n_s; s0 += 8u) {
        float4 v[8];
#pragma unroll
        for (uint32_t i = 0; i < 8u; ++i) {
            const uint32_t sidx = s0 + i;
            v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (sidx < n_s) v[i] = qmp_load_group_raw(d, places.unit(sidx), lane);
        }
#pragma unroll
        for (uint32_t i = 0; i < 8u; ++i) acc += qmp_abs_sum_raw(d.w_bf16 != 0u, v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    return acc / (static_cast<float>(n_s) * 128.0f);
}

// The loader: walks the CTA's ranges of matrix 0, 1, 2, ... stage by stage.  qmp_loader_issue starts up to
// `max_copies` copies (each after its stage has been released) and returns false if a wait ran out.
struct QmpLoader {
    int m;                       // matrix being loaded
    uint32_t u, u_end;           // next unit and end of the CTA's range of it (valid while `open`)
    uint32_t unit_bytes;
    const char* W;
    bool open;
    QmpRing ring;
    uint32_t issued;             // copies of this launch (the drain after an abort needs it)
    unsigned long long policy;   // L2 policy of the copies: read once
};
__device__ __forceinline__ bool qmp_loader_issue(QmpLoader& L, const QmpBatch& batch, int count, uint32_t max_copies,
                                                 uint32_t grid_magic, uint32_t ring_base, uint32_t bar_full0, uint32_t bar_empty0, volatile int* abort_flag) {
    for (;;) {
        while (!L.open) {
            if (L.m >= count) return true;
            const QmpDesc d = qmp_desc_of(batch, L.m);
            const QmpRange rg = qmp_range(d, grid_magic);
            L.u = rg.u_begin;
            L.u_end = rg.u_end;
            L.unit_bytes = d.w_bf16 ? 256u : 512u;
            L.W = static_cast<const char*>(d.W);
            if (L.u < L.u_end) L.open = true; else ++L.m;
        }
        if (max_copies == 0u) return true;
        --max_copies;
        if (!qmp_mbar_wait(bar_empty0 + 8u * L.ring.stage(), L.ring.phase() ^ 1u, abort_flag)) return false;
        const uint32_t units = min(L.u_end - L.u, static_cast<uint32_t>(kQmpStageBytes) / L.unit_bytes);
        const uint32_t bytes = units * L.unit_bytes;
        qmp_mbar_expect_tx(bar_full0 + 8u * L.ring.stage(), bytes);
        bulk_load_once(ring_base + L.ring.stage() * kQmpStageBytes, L.W + static_cast<size_t>(L.u) * L.unit_bytes, bytes, bar_full0 + 8u * L.ring.stage(),
                           L.policy);
        ++L.issued;
        L.ring.advance();
        L.u += units;
        if (L.u >= L.u_end) { L.open = false; ++L.m; }
    }
}

// The job of matrix d for this CTA (everything but the bracket).
__device__ __forceinline__ void qmp_make_job(const QmpDesc& d, uint32_t grid_magic, QmpJob& jb) {
    const QmpRange rg = qmp_range(d, grid_magic);
    jb.vals = reinterpret_cast<unsigned char*>(d.vals);
    jb.meta = d.meta;
    jb.prev = d.prev_meta;
    jb.KB = d.KB;
    jb.kb_magic = d.kb_magic;
    jb.units = rg.u_end - rg.u_begin;
    jb.n0 = qmp_div(rg.u_begin, d.KB, d.kb_magic, jb.kb0);
    jb.rep_n = qmp_div(kQmpStepUnits, d.KB, d.kb_magic, jb.rep_kb);
    const uint32_t next = (d.w_bf16 ? 2u * kQmpTeams - 1u : kQmpTeams) * kQmpStepUnits;     // two steps per stage of bf16 weights
    jb.next_n = qmp_div(next, d.KB, d.kb_magic, jb.next_kb);
    jb.bf16 = d.w_bf16;
}

__device__ __forceinline__ uint32_t qmp_lanes_below() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// A computing warp's list of undecided kept values; the count is the same in every lane.
struct QmpWarpList {
    QmpEntry* entries;
    uint32_t cap, n;
};
// Appends the lanes' undecided values: bit j of `und` = value j of this lane, at byte `off(j)` of vals with weight
// `value(j)`.  Whole warp.  No atomics: the lanes' places come from ballots (mostly one round: few lanes have two).
template <typename Off, typename Value>
__device__ __forceinline__ void qmp_list_append(QmpWarpList& list, uint32_t und, Off off, Value value) {
    for (uint32_t who = __ballot_sync(0xFFFFFFFFu, und != 0u); who != 0u; who = __ballot_sync(0xFFFFFFFFu, und != 0u)) {
        if (und != 0u) {
            const int j = __ffs(static_cast<int>(und)) - 1;
            const uint32_t at = list.n + __popc(who & qmp_lanes_below());
            if (at < list.cap) { list.entries[at].byte_off = off(j); list.entries[at].w = value(j); }
            und &= und - 1u;
        }
        list.n += __popc(who);
    }
}

// Mask bits that differ between two metadata words of four groups, halved: two kept pairs of a group are the same
// (xor 0), share one column (2 bits differ) or none (4); the last happens exactly for the xors 5 and 10.
__device__ __forceinline__ uint32_t qmp_flip_pairs(uint32_t x) {
    const uint32_t any = (x | (x >> 1) | (x >> 2) | (x >> 3)) & 0x11111111u;
    const uint32_t same = ~(x ^ (x >> 2));                            // bits 0 / 1 of a nibble equal its bits 2 / 3
    const uint32_t none = same & (same >> 1) & (x ^ (x >> 1)) & 0x11111111u;
    return __popc(any | (none << 1));
}

// The bracket as the computing warps use it.  fp32: a weight is kept as +-1 iff |w| > thr_pred, i.e. iff thr_pred - |w| is
// negative, and undecided iff that difference lies in 0 .. width (an unsigned compare of the bits; the subtraction is exact near
// the threshold and monotone everywhere: a value wrongly taken for undecided can only lie below the bracket, and the fix-up decides it
// like any other).  bf16 in halfword arithmetic: the largest |w| that is not above / not inside the bracket, in both halves.
template <bool BF16>
struct QmpBracket {
    float thr_pred, lo_pred;
    uint32_t width;
    uint32_t hi2, lo2;
    __device__ __forceinline__ explicit QmpBracket(const QmpJob& jb) {
        float lo, hi;
        asm volatile("ld.volatile.shared.v2.f32 {%0, %1}, [%2];" : "=f"(lo), "=f"(hi) : "r"(qmp_smem_u32(&jb.bracket)));
        const uint32_t hi_bits = __float_as_uint(hi) - 1u, lo_bits = __float_as_uint(lo) - 1u;
        thr_pred = __uint_as_float(hi_bits);
        lo_pred = __uint_as_float(lo_bits);
        width = __float_as_uint(thr_pred - lo);
        hi2 = (hi_bits >> 16) * 0x10001u;
        lo2 = (lo_bits >> 16) * 0x10001u;
    }
};

// Where a computing warp is in a matrix: its quarter-warp's unit of the current step of its team's stages.
template <bool BF16>
struct QmpWalk {
    static constexpr uint32_t kUnitBytes = BF16 ? 256u : 512u;
    static constexpr uint32_t REP = kQmpStageBytes / (kQmpStepUnits * kUnitBytes);     // steps per stage
    uint32_t n, kb;                       // row and 128-column block
    int left;                             // > 0: the quarter-warp has a unit in the step
    __device__ __forceinline__ QmpWalk(const QmpJob& jb, uint32_t stage_in_matrix, uint32_t in_step) {
        const uint32_t u0 = stage_in_matrix * (REP * kQmpStepUnits) + in_step;         // from the range's start
        n = jb.n0 + qmp_div(jb.kb0 + u0, jb.KB, jb.kb_magic, kb);
        left = static_cast<int>(jb.units) - static_cast<int>(u0);
    }
    __device__ __forceinline__ void advance(const QmpJob& jb, uint32_t KB, bool in_stage) {
        n += in_stage ? jb.rep_n : jb.next_n;
        kb += in_stage ? jb.rep_kb : jb.next_kb;
        if (kb >= KB) { kb -= KB; ++n; }
        left -= static_cast<int>((in_stage ? 1u : (kQmpTeams * REP - REP + 1u)) * kQmpStepUnits);
    }
};

// The first look: a matrix without a hint starts with a wide bracket (a sample of 64 or 256 units), and nearly every warp meets
// undecided weights in every step then -- a fifth of pass 1's time.  So the CTAs tell each other, in the same slots but under
// another tag, the mean |w| of what they have seen after their teams' first stages, and the bracket becomes as narrow as the spread of
// these means allows (five standard errors: 0.3 % for Gaussian weights).  Nobody waits for it: the finisher looks while pass 1
// runs and gives up when it has ended, and a CTA that is already done (its exchange's tag is in the slot) is left out.  Results
// never depend on the bracket.
constexpr unsigned long long kQmpLookTag = 1ull << 63;
constexpr float kQmpLookErrors = 5.0f, kQmpLookLeast = 0.001f;
// From this many units of a CTA on: shorter ranges are over before the answer is there.  With it / without, 21 sizes, light and heavy tails:
// 2:4 346 units fp32 1.09, 519 bf16 1.06, 606 1.00 to 1.02, 692 0.98 to 1.00, 934 0.95 to 0.98, 1384 0.92 to 0.94; 6:8 519 0.97 to 0.99, 692 0.95 to 0.98,
// 934 0.92 to 0.94 (2560 -> 6912 6:8 fp32 33.4 / 31.1 us).
constexpr uint32_t kQmpLookFrom = 700;
__device__ __forceinline__ void qmp_look_report(QmpStreamShared& sh, double acc) {
    float sum = static_cast<float>(acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if ((threadIdx.x & 31u) == 0u) {
        sh.look_sum[threadIdx.x >> 5] = sum;
        qmp_mbar_arrive(qmp_smem_u32(&sh.bar_look));
    }
}
__device__ __forceinline__ uint32_t qmp_look_units(uint32_t units, uint32_t bf16) {      // of a CTA's range: the first stage of each team
    return min(units, kQmpTeams * (bf16 ? 2u : 1u) * kQmpStepUnits);
}

// Pass 1 of one matrix for a computing warp: its four units of every step of its team's stages (a quarter-warp per
// unit, a lane 16 weights = four groups).  The matrix's stages are the ring's g0 .. g0 + n - 1, the team's next one is
// `next_stage`.  Returns the thread's sum |W|; `ok` turns false if a wait ran out.
//
// The instructions are what this pass costs: the memory delivers 256 weights per SM every 44 clocks (fp32), and
// selection, signs, comparisons and the fp64 sum of 256 weights alone take 24 (8 more are their shared-memory
// reads).  An earlier form with 8 weights per lane spent 231 warp instructions on them, more than half beside that
// core.  So: 16 weights per lane and step (one 8-byte store of values, one 2-byte store of metadata, one
// look at the previous metadata); the selection's predicates are folded into the compares;
// "|k| >= thr" and "is |k| undecided" come from ONE subtraction, e = pred(thr_hi) - |k| (its sign bit is the first
// answer, e <= pred(thr_hi) - thr_lo as an unsigned compare of the bits the second, and four sign bits become four
// byte masks by byte permutes); the undecided are appended with ballots instead of atomics; flips are counted
// for four groups at a time from the xor of the metadata.
//
// A lane's 64 B (fp32) are read as 16-byte pieces in rotated order, (i + l8 / 2) mod 4, so that the eight lanes of a
// unit hit different banks; the rotation is undone on the 8 + 2 result bytes (two byte permutes, one shift).
template <bool BF16, bool LOOK>
__device__ __forceinline__ double qmp_stream_pass1(const QmpJob& jb, QmpStreamShared& sh, bool look, QmpWarpList& list, unsigned int& flips, uint32_t& g0, uint32_t& next_stage,
                                                   uint32_t ring_base, uint32_t bar_full0, uint32_t bar_empty0, volatile int* abort_flag, bool& ok) {
    const int lane = threadIdx.x & 31;
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t l8 = lane & 7;
    using Walk = QmpWalk<BF16>;
    constexpr uint32_t kUnitBytes = Walk::kUnitBytes, REP = Walk::REP;
    constexpr int PIECES = BF16 ? 2 : 4;                              // 16-byte pieces per lane
    const uint32_t KB = jb.KB;
    const uint32_t n_stages = (jb.units + REP * kQmpStepUnits - 1u) / (REP * kQmpStepUnits);
    const uint32_t g_end = g0 + n_stages;
    double acc = 0.0;
    const uint32_t in_step = 4u * (warp % kQmpTeamWarps) + (lane >> 3);          // this quarter-warp's unit of every step
    Walk at(jb, next_stage - g0, in_step);
    const uint32_t turn = BF16 ? (l8 >> 2) : (l8 >> 1);               // rotation of the pieces ...
    const uint32_t rot = BF16 ? 2u * turn : turn;                     // ... and of the groups
    uint32_t src[PIECES];
#pragma unroll
    for (int i = 0; i < PIECES; ++i) src[i] = ring_base + in_step * kUnitBytes + l8 * (kUnitBytes / 8u) + 16u * ((i + turn) & (PIECES - 1u));
    // result bytes 2 p, 2 p + 1 (p = group of the unit's row) come from the group read as number (p - rot) mod 4
    uint32_t sel_lo = 0u, sel_hi = 0u;
#pragma unroll
    for (uint32_t p = 0; p < 2; ++p) {
        const uint32_t i_lo = (p - rot) & 3u, i_hi = (p + 2u - rot) & 3u;
        sel_lo |= ((2u * i_lo) | ((2u * i_lo + 1u) << 4)) << (8u * p);
        sel_hi |= ((2u * i_hi) | ((2u * i_hi + 1u) << 4)) << (8u * p);
    }
    uint8_t* const meta_lane = jb.meta + 2u * l8;
    const uint8_t* const prev_lane = jb.prev != nullptr ? jb.prev + 2u * l8 : nullptr;
    const uint32_t chunk = l8 >> 1;
    // row index in the tiled order: 16 B of metadata and 64 B of values each (layouts.cuh)
    auto tiled_row = [&](uint32_t nn, uint32_t kk) { return (((nn >> 7) * KB + kk) << 7) + (nn & 127u); };
    uint32_t q = tiled_row(at.n, at.kb);
    uint32_t prev = 0u;
    if (prev_lane != nullptr && at.left > 0) prev = *reinterpret_cast<const uint16_t*>(prev_lane + static_cast<size_t>(q) * 16u);
    QmpBracket<false> br(jb);                                         // (bf16 weights are fp32 by then)
    for (; next_stage < g_end; next_stage += kQmpTeams) {
        const uint32_t use = next_stage / kQmpStages, stage = next_stage - use * kQmpStages;
        if (!qmp_mbar_wait(bar_full0 + 8u * stage, use & 1u, abort_flag)) { ok = false; break; }
        if constexpr (LOOK) br = QmpBracket<false>(jb);               // may have become narrower
#pragma unroll
        for (uint32_t rep = 0; rep < REP; ++rep) {
            // The warp has no unit in this step (a matrix's last stage): nothing to do.  (Batch of 14 bf16 tensors 124 -> 120 us; of fp32
            // ones 130.6 without, 133.4 with it.)
            if ((BF16 || LOOK) && at.left + (lane >> 3) <= 0) {
                if (rep + 1 == REP && lane == 0) qmp_mbar_arrive(bar_empty0 + 8u * stage);
                at.advance(jb, KB, rep + 1 < REP);
                continue;
            }
            float4 raw[PIECES];
            // a lane without a unit (last stage only) reads what is there: it is not used
#pragma unroll
            for (int i = 0; i < PIECES; ++i) raw[i] = qmp_lds128(src[i] + stage * kQmpStageBytes + rep * (kQmpStepUnits * kUnitBytes));
            if (rep + 1 == REP) {
                __syncwarp();
                if (lane == 0) qmp_mbar_arrive(bar_empty0 + 8u * stage);   // the values are in registers: the stage may be refilled
            }
            const bool mine = at.left > 0;
            const uint32_t q_cur = q, prev_cur = prev;
            const uint32_t v8 = q_cur * 8u + 2u * (chunk ^ ((at.n >> 1) & 3u)) + (l8 & 1u);       // 8-byte piece of the values
            at.advance(jb, KB, rep + 1 < REP);
            q = tiled_row(at.n, at.kb);
            if (prev_lane != nullptr && at.left > 0) prev = *reinterpret_cast<const uint16_t*>(prev_lane + static_cast<size_t>(q) * 16u);
            float k[8];
            uint32_t nibbles = 0u;
            double sum = 0.0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 w;
                if constexpr (BF16) {
                    const float4 r4 = raw[i >> 1];
                    const uint32_t r0 = __float_as_uint((i & 1) ? r4.z : r4.x), r1 = __float_as_uint((i & 1) ? r4.w : r4.y);
                    w = make_float4(bf16lo_to_f32(r0), bf16hi_to_f32(r0), bf16lo_to_f32(r1), bf16hi_to_f32(r1));
                } else {
                    w = raw[i];
                }
                sum += abs_sum4(w);
                nibbles |= select_pair(w, k[2 * i], k[2 * i + 1]) << (4 * i);
            }
            const uint32_t word = ((nibbles * 0x10001u) >> (16u - 4u * rot)) & 0xFFFFu;        // nibble i to its place, (i + rot) mod 4
            uint32_t e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = __float_as_uint(br.thr_pred - fabsf(k[i]));
            uint32_t t[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t keep = sign_bytes4(e[4 * h], e[4 * h + 1], e[4 * h + 2], e[4 * h + 3]);
                t[h] = (sign_bytes4(k[4 * h], k[4 * h + 1], k[4 * h + 2], k[4 * h + 3]) | 0x01010101u) & keep;
            }
            uint32_t und = 0u;
            if (mine) {
                acc += sum;
                *reinterpret_cast<uint16_t*>(meta_lane + static_cast<size_t>(q_cur) * 16u) = static_cast<uint16_t>(word);
                *reinterpret_cast<uint2*>(jb.vals + static_cast<size_t>(v8) * 8u) = make_uint2(prmt(t[0], t[1], sel_lo), prmt(t[0], t[1], sel_hi));
                if (prev_lane != nullptr) flips += qmp_flip_pairs(word ^ prev_cur);
                if (umin8(e) <= br.width) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) und |= e[i] <= br.width ? 1u << i : 0u;
                }
            }
            qmp_list_append(list, und, [&](int j) { return v8 * 8u + 2u * (((j >> 1) + rot) & 3u) + (j & 1u); },
                            [&](int j) {
                                const float a = j & 1 ? k[1] : k[0], b = j & 1 ? k[3] : k[2], c = j & 1 ? k[5] : k[4], d = j & 1 ? k[7] : k[6];
                                return j & 4 ? (j & 2 ? d : c) : (j & 2 ? b : a);
                            });
        }
        if constexpr (LOOK) {
            if (look) { qmp_look_report(sh, acc); look = false; }
        }
    }
    if constexpr (LOOK) {
        if (look) qmp_look_report(sh, 0.0);                           // no stage of this matrix was the team's
    }
    g0 = g_end;
    flips *= 2u;
    return acc;
}

// Eight consecutive weights (half of a lane's 16): fp32 in eight words, bf16 in four.
// Sum |w| in fp64.  |bf16| becomes a double by two integer instructions (see bf16_abs_to_f64 in norm_quant_act.cuh: a zero
// counts as 2^-127, which no sum above the 1e-5 clamp can see; the sums of a lane that saw an infinity or a NaN are taken again, below);
// fp32 takes the conversion instruction.
template <bool BF16>
__device__ __forceinline__ double qmp_abs_sum8(const uint32_t* r) {
    double d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if constexpr (BF16) {
            const uint32_t w = r[i >> 1];
            d[i] = __hiloint2double(static_cast<int>(((i & 1) ? (w & 0x7FFF0000u) >> 3 : (w & 0x7FFFu) << 13) + 0x38000000u), 0);
        } else {
            d[i] = static_cast<double>(fabsf(__uint_as_float(r[i])));
        }
    }
    return ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7]));
}

// A lane's 16 bf16 weights as fp32 weights of the same values are selected and summed: for infinities and NaN, whose exponent field
// qmp_abs_sum8 takes for 2^128 (and select6of8_bf16 orders by their bits), so that a diverged run shows in the scale.
__device__ __forceinline__ void select_and_sum_as_f32(const uint32_t (&r)[8], uint32_t (&S)[2], double& sum) {
    sum = 0.0;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        float a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t w = r[4 * g + (i >> 1)];
            a[i] = fabsf((i & 1) ? bf16hi_to_f32(w) : bf16lo_to_f32(w));
            sum += static_cast<double>(a[i]);
        }
        S[g] = select6of8(a);
    }
}

// Ternary bytes of eight weights at the upper end of the bracket (t_lo, t_hi), and whether one of them may be undecided.
// Byte order: columns 0 .. 7.
template <bool BF16>
__device__ __forceinline__ void qmp_ternary8(const uint32_t* r, const QmpBracket<BF16>& br, uint32_t& t_lo, uint32_t& t_hi, bool& maybe) {
    uint32_t sign_lo, sign_hi, keep_lo, keep_hi;
    if constexpr (BF16) {
        uint32_t h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { h[i] = sub_abs_bf16x2(br.hi2, r[i]); l[i] = sub_abs_bf16x2(br.lo2, r[i]); }
        const uint32_t open = ((l[0] & ~h[0]) | (l[1] & ~h[1])) | ((l[2] & ~h[2]) | (l[3] & ~h[3]));
        keep_lo = prmt(h[0], h[1], kSign2); keep_hi = prmt(h[2], h[3], kSign2);
        sign_lo = prmt(r[0], r[1], kSign2); sign_hi = prmt(r[2], r[3], kSign2);
        maybe |= (open & kGuard2) != 0u;
    } else {
        uint32_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = __float_as_uint(br.thr_pred - fabsf(__uint_as_float(r[i])));
        keep_lo = sign_bytes4(e[0], e[1], e[2], e[3]); keep_hi = sign_bytes4(e[4], e[5], e[6], e[7]);
        sign_lo = sign_bytes4(r[0], r[1], r[2], r[3]); sign_hi = sign_bytes4(r[4], r[5], r[6], r[7]);
        maybe |= umin8(e) <= br.width;
    }
    t_lo = (sign_lo | 0x01010101u) & keep_lo;
    t_hi = (sign_hi | 0x01010101u) & keep_hi;
}
// Byte masks of the undecided ones among them: inside the bracket and not kept as +-1.
template <bool BF16>
__device__ __forceinline__ void qmp_undecided8(const uint32_t* r, const QmpBracket<BF16>& br, uint32_t t_lo, uint32_t t_hi, uint32_t& u_lo, uint32_t& u_hi) {
    if constexpr (BF16) {
        uint32_t g[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) g[i] = sub_abs_bf16x2(br.lo2, r[i]);
        u_lo = prmt(g[0], g[1], kSign2); u_hi = prmt(g[2], g[3], kSign2);
    } else {
        uint32_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = __float_as_uint(br.lo_pred - fabsf(__uint_as_float(r[i])));
        u_lo = sign_bytes4(e[0], e[1], e[2], e[3]); u_hi = sign_bytes4(e[4], e[5], e[6], e[7]);
    }
    u_lo &= ~((t_lo & 0x01010101u) * 0xFFu);                          // a byte of t is 0, 1 or 0xFF
    u_hi &= ~((t_hi & 0x01010101u) * 0xFFu);
}

template <bool BF16>
__device__ __forceinline__ float qmp_lds_weight(uint32_t addr) {
    if constexpr (BF16) {
        uint16_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
        return __uint_as_float(static_cast<uint32_t>(v) << 16);
    } else {
        float v;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
        return v;
    }
}

// Reads the 16 weights of a lane: eight words of bf16 or sixteen of fp32, in 16-byte pieces from src[i] + off.
template <int PIECES>
__device__ __forceinline__ void qmp_lds_pieces(const uint32_t (&src)[PIECES], uint32_t off, uint32_t (&r)[4 * PIECES]) {
#pragma unroll
    for (int i = 0; i < PIECES; ++i)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[4 * i]), "=r"(r[4 * i + 1]), "=r"(r[4 * i + 2]), "=r"(r[4 * i + 3]) : "r"(src[i] + off));
}

// Pass 1 for the 6:8 pattern.  As above; a lane's 16 weights are two groups of 8, which leave as 12 value bytes (three 4-byte
// stores) and 24 bits of metadata (a quad of lanes has 12 bytes, its lanes 0..2 store 4 each).  The two groups are read in the
// order that halves the bank conflicts of the 64 B (fp32; none for bf16) per lane and put in place on the results.
//
// The ALU pipe (byte permutes, logic, minima: half rate) bounds it, so comparisons are subtractions on the FMA pipe whose sign bits
// are gathered by byte permutes, and bf16 weights are selected two to a word.  The undecided are looked for only if one of the
// warp's weights lies inside the bracket, for both groups at once, and their weights come from the stage again (held until then) instead of
// a tree of selects.  Single calls without a hint, us, before / now (with the loops over matrices gone and the first look):
// 2560 -> 2560 fp32 20.8 / 17.0, 2560 -> 6912 fp32 36.9 / 30.7, bf16 38.2 / 27.9 (memory: 13.5 and 8.1).
template <bool BF16>
__device__ __forceinline__ double qmp68_stream_pass1(const QmpJob& jb, QmpStreamShared& sh, bool look, QmpWarpList& list, unsigned int& flips, uint32_t& g0, uint32_t& next_stage,
                                                     uint32_t ring_base, uint32_t bar_full0, uint32_t bar_empty0, volatile int* abort_flag, bool& ok,
                                                     const uint2* table) {
    const int lane = threadIdx.x & 31;
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t l8 = lane & 7, quad = l8 & 3u;
    using Walk = QmpWalk<BF16>;
    constexpr uint32_t kUnitBytes = Walk::kUnitBytes, REP = Walk::REP;
    constexpr int PIECES = BF16 ? 2 : 4;
    const uint32_t KB = jb.KB, KBp = KB + (KB >> 1);                  // K' / 128
    const uint32_t g_end = g0 + (jb.units + REP * kQmpStepUnits - 1u) / (REP * kQmpStepUnits);
    double acc = 0.0;
    const uint32_t in_step = 4u * (warp % kQmpTeamWarps) + (lane >> 3);
    Walk at(jb, next_stage - g0, in_step);
    const uint32_t swap = BF16 ? (l8 >> 2) : ((l8 >> 1) & 1u);        // the second group is read first
    const uint32_t src0 = ring_base + in_step * kUnitBytes + l8 * (kUnitBytes / 8u);
    uint32_t src[PIECES];
#pragma unroll
    for (int i = 0; i < PIECES; ++i) src[i] = src0 + 16u * (static_cast<uint32_t>(i) ^ (swap * (PIECES / 2)));
    // Column block kb of a row starts at byte 96 kb of its values and 24 kb of its metadata in the [N][K'] form: in tile 3 kb / 2,
    // for odd kb half a tile in.  With q = the row's index in that tile, a lane's three words of values are at
    // 64 q + (v ^ the row's swizzle) and its word of its quad's metadata at 16 q + m, v and m constants for even
    // (low half) and odd (high half) kb.
    auto tiled_row = [&](uint32_t nn, uint32_t kk) { return (((nn >> 7) * KBp + ((3u * kk) >> 1)) << 7) + (nn & 127u); };
    uint32_t v_const[3], m_const = 0u;
#pragma unroll
    for (uint32_t odd = 0; odd < 2; ++odd) {
#pragma unroll
        for (uint32_t i = 0; i < 3; ++i) {
            const uint32_t y = 12u * l8 + 4u * i + 32u * odd;
            v_const[i] = (odd ? v_const[i] : 0u) | (((y >> 6) * 8192u + (y & 63u)) << (16u * odd));
        }
        const uint32_t y = 12u * (l8 >> 2) + 4u * quad + 8u * odd;
        m_const |= ((y >> 4) * 2048u + (y & 15u)) << (16u * odd);
    }
    const bool has_prev = jb.prev != nullptr;
    uint32_t q = tiled_row(at.n, at.kb), prev = 0u;
    auto meta_at = [&](uint32_t qq, uint32_t kk) { return static_cast<size_t>(qq) * 16u + ((kk & 1u) ? m_const >> 16 : m_const & 0xFFFFu); };
    if (has_prev && quad < 3u && at.left > 0) prev = *reinterpret_cast<const uint32_t*>(jb.prev + meta_at(q, at.kb));
    for (; next_stage < g_end; next_stage += kQmpTeams) {
        const uint32_t use = next_stage / kQmpStages, stage = next_stage - use * kQmpStages;
        if (!qmp_mbar_wait(bar_full0 + 8u * stage, use & 1u, abort_flag)) { ok = false; break; }
        const QmpBracket<BF16> br(jb);                                // may have become narrower
#pragma unroll 1
        for (uint32_t rep = 0; rep < REP; ++rep) {
            if (at.left + (lane >> 3) <= 0) {                         // the warp has no unit in this step (a matrix's last stage)
                at.advance(jb, KB, rep + 1 < REP);
                continue;
            }
            uint32_t r[4 * PIECES];
            const uint32_t off = stage * kQmpStageBytes + rep * (kQmpStepUnits * kUnitBytes);
            qmp_lds_pieces(src, off, r);
            const bool mine = at.left > 0;
            const uint32_t q_cur = q, odd_cur = at.kb & 1u, prev_cur = prev;
            const uint32_t half = odd_cur ? 0x4432u : 0x4410u, swizzle = ((at.n >> 1) & 3u) << 4;
            at.advance(jb, KB, rep + 1 < REP);
            q = tiled_row(at.n, at.kb);
            if (has_prev && quad < 3u && at.left > 0) prev = *reinterpret_cast<const uint32_t*>(jb.prev + meta_at(q, at.kb));
            auto v_off = [&](uint32_t v) { return prmt(v, 0u, half) ^ swizzle; };           // on top of 64 q_cur
            constexpr int kHalf = 2 * PIECES;                         // words of a group
            uint32_t S[2];
            double sum = qmp_abs_sum8<BF16>(r) + qmp_abs_sum8<BF16>(r + kHalf);
            if constexpr (BF16) {
                select6of8_bf16(r, S[0], S[1]);
                if (__double2hiint(sum) >= 0x47F00000) select_and_sum_as_f32(r, S, sum);      // 2^128 or more
            } else {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    float a[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) a[i] = fabsf(__uint_as_float(r[8 * g + i]));
                    S[g] = select6of8(a);
                }
            }
            uint2 entry[2];
            uint32_t t_lo[2], t_hi[2], v4[2], v2[2];
            bool maybe = false;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                entry[g] = table[S[g]];
                qmp_ternary8<BF16>(r + kHalf * g, br, t_lo[g], t_hi[g], maybe);
                v4[g] = prmt(t_lo[g], t_hi[g], entry[g].x);
                v2[g] = prmt(t_lo[g], t_hi[g], entry[g].x >> 16);     // two bytes
            }
            const uint32_t f4 = swap ? v4[1] : v4[0], f2 = swap ? v2[1] : v2[0], l4 = swap ? v4[0] : v4[1], l2 = swap ? v2[0] : v2[1];
            const uint32_t m24 = swap ? (entry[1].y | (entry[0].y << 12)) : (entry[0].y | (entry[1].y << 12));
            const uint32_t nxt = __shfl_down_sync(0xFFFFFFFFu, m24, 1);
            if (has_prev) {
                // this lane's 24 bits of the previous metadata, from its own and the lane before's word
                const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, prev_cur, 1);
                const uint32_t p24 = (quad == 0u ? prev_cur : ((before >> (32u - 8u * quad)) | (prev_cur << (8u * quad)))) & 0xFFFFFFu;
                if (mine && p24 != m24)
                    flips += __popc((swap ? S[1] : S[0]) ^ mask8_from_meta12(p24)) + __popc((swap ? S[0] : S[1]) ^ mask8_from_meta12(p24 >> 12));
            }
            if (mine) {
                acc += sum;
                if (quad < 3u) *reinterpret_cast<uint32_t*>(jb.meta + meta_at(q_cur, odd_cur)) = (m24 >> (8u * quad)) | (nxt << (24u - 8u * quad));
                unsigned char* const row = jb.vals + static_cast<size_t>(q_cur) * 64u;
                *reinterpret_cast<uint32_t*>(row + v_off(v_const[0])) = f4;
                *reinterpret_cast<uint32_t*>(row + v_off(v_const[1])) = prmt(f2, l4, 0x5410u);
                *reinterpret_cast<uint32_t*>(row + v_off(v_const[2])) = prmt(l4, l2, 0x5432u);
            }
            if (__any_sync(0xFFFFFFFFu, mine && maybe)) {
                uint32_t und = 0u;
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    uint32_t u_lo, u_hi;
                    qmp_undecided8<BF16>(r + kHalf * g, br, t_lo[g], t_hi[g], u_lo, u_hi);
                    und |= (qmp_byte_bits(u_lo, u_hi) & S[g]) << (8 * g);
                }
                qmp_list_append(list, mine ? und : 0u,
                                [&](int j) {                          // column j & 7 of the group read as number j >> 3
                                    const uint32_t g = static_cast<uint32_t>(j) >> 3;
                                    const uint32_t at_byte = 6u * (g ^ swap) + __popc((g ? S[1] : S[0]) & ((1u << (j & 7)) - 1u));   // of the lane's 12
                                    return q_cur * 64u + v_off(at_byte < 4u ? v_const[0] : (at_byte < 8u ? v_const[1] : v_const[2])) + (at_byte & 3u);
                                },
                                [&](int j) {
                                    const uint32_t g = (static_cast<uint32_t>(j) >> 3) ^ swap;
                                    return qmp_lds_weight<BF16>(src0 + off + g * (kUnitBytes / 16u) + (j & 7) * (kUnitBytes / 128u));
                                });
            }
        }
        __syncwarp();
        if (lane == 0) qmp_mbar_arrive(bar_empty0 + 8u * stage);      // the stage may be refilled
        if (look) { qmp_look_report(sh, acc); look = false; }
    }
    if (look) qmp_look_report(sh, 0.0);
    g0 = g_end;
    return acc;
}

// {tag, partial sum} of a CTA as one 128-bit word: whoever sees the tag has the sum (no fence, one trip).
__device__ __forceinline__ void qmp_slot_store(QmpSlot* slot, unsigned long long tag, double partial) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}"
                 ::"l"(slot), "l"(tag), "l"(__double_as_longlong(partial)) : "memory");
}
__device__ __forceinline__ unsigned long long qmp_slot_peek(const QmpSlot* slot, double& partial) {
    unsigned long long t;
    long long v;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(t), "=l"(v) : "l"(slot) : "memory");
    partial = __longlong_as_double(v);
    return t;
}
__device__ __forceinline__ bool qmp_slot_load(const QmpSlot* slot, unsigned long long tag, double& partial) {
    double v;
    if (qmp_slot_peek(slot, v) != tag) return false;
    partial = v;
    return true;
}

// The sum of all CTAs' partial sums of a matrix by one warp, in a fixed order: the same bits in every CTA.  A lane
// looks after the slots lane, lane + 32, ..., all of them polled together.  False if the wait ran out.
__device__ __forceinline__ bool qmp_exchange(const QmpSlot* base, unsigned long long tag, int lane, volatile int* abort_flag, double& sum) {
    constexpr int kPerLane = (kQmpMaxCtas + 31) / 32;
    double part[kPerLane];
    uint32_t missing = 0u;
#pragma unroll
    for (int j = 0; j < kPerLane; ++j) {
        part[j] = 0.0;
        if (lane + 32u * j < gridDim.x) missing |= 1u << j;
    }
    unsigned long long t0 = 0ull;
    unsigned int spins = 0;
    bool ok = true;
    while (missing != 0u) {
#pragma unroll
        for (int j = 0; j < kPerLane; ++j)
            if (((missing >> j) & 1u) != 0u && qmp_slot_load(&base[lane + 32 * j], tag, part[j])) missing &= ~(1u << j);
        if (missing != 0u && ((++spins & 0xFFu) == 0u)) {
            if (*abort_flag) { ok = false; break; }
            const unsigned long long now = global_timer_ns_qmp();
            if (t0 == 0ull) t0 = now;
            else if (now - t0 > *reinterpret_cast<volatile unsigned long long*>(&g_wait_limit_ns)) { ok = false; break; }
        }
    }
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok) {
        if (lane == 0) { *abort_flag = 1; atomicExch(&g_device_status, static_cast<int>(SBN_ERR_TIMEOUT)); }
        return false;
    }
    sum = 0.0;
#pragma unroll
    for (int j = 0; j < kPerLane; ++j) sum += part[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    return true;
}

// The first look, by the finisher (see qmp_look_report).  Returns when the bracket has been narrowed or pass 1 of matrix 0 is over.
__device__ __forceinline__ bool qmp_look_exchange(const QmpDesc& first, QmpStreamShared& sh, QmpSlot* slots, unsigned long long tag, int lane, volatile int* abort_flag) {
    if (!qmp_mbar_wait(qmp_smem_u32(&sh.bar_look), 0u, abort_flag)) return false;
    QmpJob& jb = sh.job[0];
    const uint32_t seen = qmp_look_units(jb.units, jb.bf16), bar_done = qmp_smem_u32(&sh.bar_done[0]);
    float sum = lane < kQmpStreamWarps ? sh.look_sum[lane] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if (lane == 0) qmp_slot_store(slots + blockIdx.x, tag ^ kQmpLookTag, seen != 0u ? static_cast<double>(sum / (128.0f * static_cast<float>(seen))) : -1.0);
    __syncwarp();
    constexpr int kPerLane = (kQmpMaxCtas + 31) / 32;
    uint32_t missing = 0u;
    float n = 0.0f, s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int j = 0; j < kPerLane; ++j)
        if (lane + 32u * j < gridDim.x) missing |= 1u << j;
    while (__any_sync(0xFFFFFFFFu, missing != 0u)) {
        if (__any_sync(0xFFFFFFFFu, qmp_mbar_try_wait(bar_done, 0u) || *abort_flag != 0)) return true;      // pass 1 has ended (or will not): too late
#pragma unroll
        for (int j = 0; j < kPerLane; ++j) {
            double mean;
            if (((missing >> j) & 1u) != 0u) {
                const unsigned long long got = qmp_slot_peek(&slots[lane + 32 * j], mean);
                if (got == tag || got == (tag ^ kQmpLookTag)) missing &= ~(1u << j);
                if (got == (tag ^ kQmpLookTag) && mean > 0.0) { const float v = static_cast<float>(mean); n += 1.0f; s1 += v; s2 += v * v; }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n += __shfl_xor_sync(0xFFFFFFFFu, n, o);
        s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
        s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
    }
    const float gamma = s1 / n, error = sqrtf(fmaxf(s2 / n - gamma * gamma, 0.0f) / n) / gamma, b = kQmpLookErrors * error + kQmpLookLeast;
    if (lane == 0 && n >= 32.0f && b > 0.0f && b < kQmpBracketSmall) {
        const float2 wide = jb.bracket, narrow = qmp_bracket(gamma, b);
        const float lo = fmaxf(wide.x, narrow.x), hi = fminf(wide.y, narrow.y);
        // outside what pass 1 has used so far: the exact threshold will miss one of the two, or the sample was far off
        if (lo < hi) asm volatile("st.volatile.shared.v2.f32 [%0], {%1, %2};" ::"r"(qmp_smem_u32(&jb.bracket)), "f"(lo), "f"(hi) : "memory");
    }
    __syncwarp();
    return true;
}

// ternary_threshold by a whole warp: lane i tries the i-th float from 8 below scale / 2, the lowest that passes is it.
__device__ __forceinline__ float qmp_threshold_warp(float scale, int lane) {
    const float a = __uint_as_float(__float_as_uint(0.5f * scale) - 8u + lane);
    const uint32_t passes = __ballot_sync(0xFFFFFFFFu, __fdiv_rn(a, scale) > 0.5f);
    return __shfl_sync(0xFFFFFFFFu, a, __ffs(static_cast<int>(passes)) - 1);
}

// Do the listed values suffice, or must the whole range be ternarised again with the exact threshold?
template <int PATTERN>
__device__ __forceinline__ bool qmp_bracket_holds(const QmpDesc& d, float thr, const QmpJob& jb, unsigned int longest_list, uint32_t list_cap) {
    return jb.bracket.x <= thr && thr <= jb.bracket.y && longest_list <= list_cap && d.dense_q == nullptr &&
           d.num_units <= (PATTERN == 68 ? 1u << 25 : 1u << 26);     // listed byte offsets are 32-bit
}
__device__ __forceinline__ void qmp_fix_entry(uint8_t* vals, const QmpEntry e, float thr) {
    vals[e.byte_off] = static_cast<uint8_t>(fabsf(e.w) >= thr ? (e.w < 0.0f ? 0xFFu : 0x01u) : 0u);
}

// Ternarises this CTA's range of matrix d again with the exact threshold.
template <int PATTERN>
__device__ __forceinline__ void qmp_second_pass(const QmpDesc& d, uint32_t grid_magic, float thr, const uint2* table) {
    const QmpRange rg = qmp_range(d, grid_magic);
    if constexpr (PATTERN == 68) {
        if (d.w_bf16) qmp68_pass2_full<true>(d, rg, thr, table);
        else qmp68_pass2_full<false>(d, rg, thr, table);
    } else {
        if (d.w_bf16) qmp_pass2_full<true>(d, rg, thr);
        else qmp_pass2_full<false>(d, rg, thr);
    }
}

// PATTERN: 24 (2:4) or 68 (6:8).  SINGLE: one matrix, known at compile time.  Without the loops over matrices a call is 1 to 2 us
// shorter; the first look would cost a batch 1 %.  Single calls without a hint, us, before / now, with 20 computing warps: 2560 ->
// 2560 fp32 17.4 / 14.9, bf16 16.9 / 13.6; 2560 -> 6912 26.5 / 23.0 and 25.3 / 21.3; 4096 -> 11008 50 / 43.6 and 46 / 39.0.
template <int PATTERN, bool SINGLE>
__global__ void __launch_bounds__(kQmpThreads, 1)
quantize_mask_pack_stream_kernel(const __grid_constant__ QmpInlineDescs inl, const QmpDesc* __restrict__ rest, int n_matrices,
                                 QmpSlot* slots, unsigned long long* generation, unsigned long long call_nonce,
                                 int test_withhold_slot, QmpMemo* memo, uint32_t grid_magic) {
    const int count = SINGLE ? 1 : n_matrices;
    extern __shared__ __align__(128) unsigned char s_dyn[];   // [kQmpStages][kQmpStageBytes] ring, then kQmpLists * kQmpListEntries entries
    QmpEntry* const s_list = reinterpret_cast<QmpEntry*>(s_dyn + kQmpStages * kQmpStageBytes);
    const uint32_t list_cap = qmp_list_cap(count);
    auto list_of = [&](int slot, int w) { return s_list + static_cast<uint32_t>(slot * kQmpStreamWarps + w) * list_cap; };
    __shared__ QmpStreamShared sh;
    __shared__ uint2 s_table[PATTERN == 68 ? 256 : 1];        // by kept set (6:8)

    const QmpBatch batch{inl, rest};
    const QmpDesc& first = inl.d[0];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    volatile int* const abort_flag = &sh.abort;
    const uint32_t ring_base = qmp_smem_u32(s_dyn);
    const uint32_t bar_full0 = qmp_smem_u32(&sh.bar_full[0]), bar_empty0 = qmp_smem_u32(&sh.bar_empty[0]);
    const uint32_t bar_done0 = qmp_smem_u32(&sh.bar_done[0]);
    if (threadIdx.x == 0) {
        sh.fixed_upto = 0;
        sh.abort = 0;
        sh.tail_second_pass = 0;
        sh.ring_issued = 0u; sh.ring_used = 0u;
        for (int i = 0; i < kQmpJobs; ++i) sh.job[i].ready = 0;
        for (int i = 0; i < kQmpLists; ++i) qmp_mbar_init(bar_done0 + 8u * i, kQmpStreamWarps);
        qmp_mbar_init(qmp_smem_u32(&sh.bar_look), kQmpStreamWarps);
        for (int i = 0; i < kQmpStages; ++i) {
            qmp_mbar_init(bar_full0 + 8u * i, 1u);                     // the loader's expect_tx
            qmp_mbar_init(bar_empty0 + 8u * i, kQmpTeamWarps);         // one arrival per computing warp of the stage's team
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 32) qmp_make_job(first, grid_magic, sh.job[0]);
    for (int i = threadIdx.x; i < count; i += kQmpThreads) sh.thr_second_pass[i] = -1.0f;
    if (PATTERN == 68 && threadIdx.x < 256) s_table[threadIdx.x] = table68_entry(threadIdx.x);
    __syncthreads();
    // No early signal to the next kernel of the stream: this kernel writes packed weights, and the
    // GEMM kernels fetch weights before their own dependency wait (see sbn_common.cuh).
    pdl_wait();

    // ---- What the first bracket needs is asked for BEFORE the loader fills the ring: the hint of matrix 0 (a 4-byte
    // read), or without a hint of the caller's its sample (all threads, one round trip) together with what an
    // earlier call may have left.  A stage per team follows at once, the rest of the ring when the bracket is known: behind all
    // stages (18 MB that the loaders of all CTAs ask for at the same moment) the sample of some CTAs comes late (single calls without a
    // hint, us, all / half the ring / a stage per team: 2560 -> 3840 fp32 18.9 / 17.0 / 16.8, bf16 17.8 / 16.0 / 15.9).
    float gamma0 = first.gamma_hint != nullptr ? *reinterpret_cast<const volatile float*>(first.gamma_hint) : 0.0f;
    float4 sample0[kQmpSamplePerWarp];
    const bool sample_early = first.gamma_hint == nullptr;
    if (sample_early) {
        unsigned long long m_tag = 0ull, m_w = 0ull;
        uint32_t m_units = 0u, m_scale = 0u;
        if (memo != nullptr) {
            // a single matrix without a hint: what the previous call on this workspace left, if it was this matrix
            asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(m_tag), "=l"(m_w) : "l"(memo));
            asm volatile("ld.volatile.global.v2.u32 {%0, %1}, [%2];" : "=r"(m_units), "=r"(m_scale) : "l"(&memo->num_units));
        }
        qmp_sample_issue(first, sample0);
        if (m_tag == kQmpMemoMagic && m_w == reinterpret_cast<unsigned long long>(first.W) && m_units == first.num_units)
            gamma0 = __uint_as_float(m_scale);
    }
    const bool hinted0 = qmp_hint_usable(gamma0);
    if (!sample_early && !hinted0) qmp_sample_issue(first, sample0);
    QmpLoader loader{0, 0u, 0u, 0u, nullptr, false, QmpRing{0u}, 0u, l2_policy_evict_first()};
    const bool is_loader = warp == kQmpLoaderWarp && lane == 0;
    if (is_loader) qmp_loader_issue(loader, batch, count, kQmpTeams, grid_magic, ring_base, bar_full0, bar_empty0, abort_flag);
    if (!hinted0) gamma0 = qmp_sample_finish(first, sample0, sh.sample);
    if (threadIdx.x == 0) {
        sh.job[0].bracket = qmp_bracket_from(gamma0, first.num_units, hinted0);
        sh.job[0].ready = 1;
        sh.look = !SINGLE || hinted0 || sh.job[0].units < kQmpLookFrom ? 0 : 1;
        if (blockIdx.x == 0 && first.flip_bits != nullptr) *first.flip_bits = 0ull;      // published with this CTA's first slot
    }
    __syncthreads();

    if (warp < kQmpStreamWarps) {
        // ------------------------------------------------------------------ computing warps
        uint32_t stages = 0u;                                // of the matrices so far
        uint32_t next_stage = static_cast<uint32_t>(warp) / kQmpTeamWarps;       // this team's
        for (int m = 0; m < count; ++m) {
            const int slot = m % kQmpLists;
            const QmpJob& jb = sh.job[m & (kQmpJobs - 1)];
            if (!qmp_wait_ge(const_cast<int*>(&jb.ready), m + 1, abort_flag)) break;
            if (!qmp_wait_ge(&sh.fixed_upto, m - (kQmpLists - 1), abort_flag)) break;
            __threadfence_block();
            unsigned int flips = 0;
            bool ok = true;
            QmpWarpList list{list_of(slot, warp), list_cap, 0u};
            double mine;
            if constexpr (PATTERN == 68)
                mine = jb.bf16 ? qmp68_stream_pass1<true>(jb, sh, SINGLE && sh.look != 0, list, flips, stages, next_stage, ring_base, bar_full0, bar_empty0, abort_flag, ok, s_table)
                               : qmp68_stream_pass1<false>(jb, sh, SINGLE && sh.look != 0, list, flips, stages, next_stage, ring_base, bar_full0, bar_empty0, abort_flag, ok, s_table);
            else
                mine = jb.bf16 ? qmp_stream_pass1<true, SINGLE>(jb, sh, SINGLE && sh.look != 0, list, flips, stages, next_stage, ring_base, bar_full0, bar_empty0, abort_flag, ok)
                               : qmp_stream_pass1<false, SINGLE>(jb, sh, SINGLE && sh.look != 0, list, flips, stages, next_stage, ring_base, bar_full0, bar_empty0, abort_flag, ok);
            if (!ok) break;
            mine += __shfl_xor_sync(0xFFFFFFFFu, mine, 16);
            mine += __shfl_xor_sync(0xFFFFFFFFu, mine, 8);
            if (lane < 8) sh.warp_sum[slot][warp][lane] = mine;
            if (jb.prev != nullptr) flips = __reduce_add_sync(0xFFFFFFFFu, flips);
            if (lane == 0) {
                sh.warp_flips[slot][warp] = flips;
                sh.warp_listed[slot][warp] = list.n;
            }
            __syncwarp();                                    // every lane's list entries and sums are written
            if (lane == 0) qmp_mbar_arrive(bar_done0 + 8u * slot);               // release: all of it before the count
        }
    } else if (warp == kQmpLoaderWarp) {
        // ------------------------------------------------------------------ the loader (one lane)
        if (is_loader) {
            qmp_loader_issue(loader, batch, count, 0xFFFFFFFFu, grid_magic, ring_base, bar_full0, bar_empty0, abort_flag);
            sh.ring_issued = loader.issued;                  // for the drain, should the CTA abort
            sh.ring_used = loader.ring.used;
        }
        __syncwarp();
    } else if (warp >= kQmpScoutWarp) {
        // ------------------------------------------------------------------ the scouts
        for (int m = 1 + (warp - kQmpScoutWarp); m < count; m += kQmpScouts) {
            const QmpDesc d = qmp_desc_of(batch, m);
            float g;
            const bool hinted = qmp_hint(d, g);
            if (!hinted) g = qmp_sample_gamma_warp(d, lane);
            // the job's place: matrix m - kQmpJobs is finished
            if (!qmp_wait_ge(&sh.fixed_upto, m - (kQmpJobs - 1), abort_flag)) break;
            if (lane == 0) {
                // zeroed well before any CTA can add to it (they add once they have seen this CTA's slot)
                if (blockIdx.x == 0 && d.flip_bits != nullptr) { *d.flip_bits = 0ull; __threadfence(); }
                QmpJob& jb = sh.job[m & (kQmpJobs - 1)];
                qmp_make_job(d, grid_magic, jb);
                jb.bracket = qmp_bracket_from(g, d.num_units, hinted, true);
                __threadfence_block();
                *reinterpret_cast<volatile int*>(&jb.ready) = m + 1;
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------------ the finisher
        const unsigned long long gen0 = *reinterpret_cast<volatile unsigned long long*>(generation);
        const unsigned long long tag = qmp_tag(call_nonce, gen0);
        bool ok = !SINGLE || sh.look == 0 || qmp_look_exchange(first, sh, slots, tag, lane, abort_flag);
        // step m: publish matrix m, then exchange and finish matrix m - 1; step `count` finishes the last matrix
        // (its fix-up is left to all warps)
        unsigned int flips_prev = 0u;
        QmpDesc dp = first;                                  // of matrix m - 1
        for (int m = 0; ok && m <= count; ++m) {
            unsigned int flips_cur = 0u;
            QmpDesc d = dp;
            if (m < count) {
                // matrix m: every computing warp has arrived -> this CTA's partial sum, published
                const int slot = m % kQmpLists;
                if (m > 0) d = qmp_desc_of(batch, m);        // on its way while the warps are waited for
                if (!qmp_mbar_wait(bar_done0 + 8u * slot, static_cast<uint32_t>(m / kQmpLists) & 1u, abort_flag)) { ok = false; break; }
                double v = 0.0;
#pragma unroll
                for (int i = 0; i < 8 * kQmpStreamWarps / 32; ++i) v += (&sh.warp_sum[slot][0][0])[lane + 32 * i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
                if (lane == 0) {
                    if (blockIdx.x == 0 && d.flip_bits != nullptr) __threadfence();      // the zeroed flip count before the slot
                    if (!(test_withhold_slot && blockIdx.x == gridDim.x - 1))
                        qmp_slot_store(slots + static_cast<size_t>(m) * gridDim.x + blockIdx.x, tag, v);
                }
                if (d.flip_bits != nullptr) flips_cur = __reduce_add_sync(0xFFFFFFFFu, lane < kQmpStreamWarps ? sh.warp_flips[slot][lane] : 0u);
                __syncwarp();
            }
            // matrix m - 1: exchange, exact threshold, fix-up
            if (m >= 1) {
                const int pslot = (m - 1) % kQmpLists;
                double sum;
                ok = qmp_exchange(slots + static_cast<size_t>(m - 1) * gridDim.x, tag, lane, abort_flag, sum);
                if (!ok) break;
                const float gamma = static_cast<float>(sum / (static_cast<double>(dp.num_units) * 128.0));
                const float scale = fmaxf(gamma, kEps);
                const float thr = qmp_threshold_warp(scale, lane);
                const unsigned int mine = lane < kQmpStreamWarps ? sh.warp_listed[pslot][lane] : 0u;     // of warp `lane`'s list
                const unsigned int longest = __reduce_max_sync(0xFFFFFFFFu, mine);
                const bool holds = qmp_bracket_holds<PATTERN>(dp, thr, sh.job[(m - 1) & (kQmpJobs - 1)], longest, list_cap);
                uint8_t* const vb = reinterpret_cast<uint8_t*>(dp.vals);
                if (m == count) {
                    if (lane == 0) { sh.thr_tail = thr; sh.tail_second_pass = holds ? 0 : 1; }
                } else if (!holds) {
                    if (lane == 0) sh.thr_second_pass[m - 1] = thr;
                } else if (longest <= 16u) {
                    // short lists (a hint): a lane per list
                    for (unsigned int i = 0; i < mine; ++i) qmp_fix_entry(vb, list_of(pslot, lane)[i], thr);
                } else {
                    for (int w = 0; w < kQmpStreamWarps; ++w) {
                        const unsigned int listed = __shfl_sync(0xFFFFFFFFu, mine, w);
                        for (unsigned int i = lane; i < listed; i += 32u) qmp_fix_entry(vb, list_of(pslot, w)[i], thr);
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    *reinterpret_cast<volatile int*>(&sh.fixed_upto) = m;
                    if (blockIdx.x == 0) *dp.w_scale = scale;
                    if (dp.flip_bits != nullptr && flips_prev != 0u) {
                        __threadfence();                     // after CTA 0's zero: its slot has been seen
                        atomicAdd(dp.flip_bits, static_cast<unsigned long long>(flips_prev));
                    }
                }
                __syncwarp();
            }
            flips_prev = flips_cur;
            dp = d;
        }
        if (ok && blockIdx.x == 0 && lane == 0) {
            // CTA 0 has read the last slots of all CTAs, so all of them have read the generation and the memo
            *reinterpret_cast<volatile unsigned long long*>(generation) = gen0 + 1ull;
            if (memo != nullptr) {
                memo->W = first.W;
                memo->num_units = first.num_units;
                memo->scale = *reinterpret_cast<volatile float*>(first.w_scale);     // written by this thread above
                __threadfence();
                memo->magic = kQmpMemoMagic;
            }
        }
    }
    __syncthreads();
    if (sh.abort) {
        // No bulk copy may still be writing this CTA's shared memory when it leaves: the last
        // min(issued, kQmpStages) copies are the ones that can be in flight; the ring position points past the newest.
        if (threadIdx.x == 0) {
            QmpRing ring{sh.ring_used};
            const uint32_t back = min(sh.ring_issued, static_cast<uint32_t>(kQmpStages));
            for (uint32_t j = 0; j < back; ++j) {
                --ring.used;
                qmp_mbar_wait(bar_full0 + 8u * ring.stage(), ring.phase(), abort_flag, true);
            }
        }
        return;
    }

    // ---- tail: fix-up (or second pass) of the last matrix, all warps; then the second passes that were put off
    {
        const int m = count - 1;
        const int slot = m % kQmpLists;
        const float thr = sh.thr_tail;
        if (sh.tail_second_pass == 0) {
            if (warp < kQmpStreamWarps) {
                uint8_t* vb = sh.job[m & (kQmpJobs - 1)].vals;
                const QmpEntry* list = list_of(slot, warp);
                const unsigned int listed = sh.warp_listed[slot][warp];
                for (unsigned int i = lane; i < listed; i += 32u) qmp_fix_entry(vb, list[i], thr);
            }
        } else {
            const QmpDesc d = qmp_desc_of(batch, m);
            qmp_second_pass<PATTERN>(d, grid_magic, thr, s_table);
        }
    }
    for (int m = 0; m + 1 < count; ++m) {
        const float thr = sh.thr_second_pass[m];
        if (thr >= 0.0f) {
            const QmpDesc d = qmp_desc_of(batch, m);
            qmp_second_pass<PATTERN>(d, grid_magic, thr, s_table);
        }
    }
}

// Launch for `count` (<= kQmpMaxBatch) matrices: the first kQmpInlineDescs of `descs_host` by value, matrices
// 1, 2, ... already copied to `rest_dev` if there are more than that.
template <int PATTERN, bool SINGLE>
inline sbn_status launch_quantize_mask_pack_stream_cfg(const QmpDesc* descs_host, const QmpDesc* rest_dev, int count,
                                                   uint32_t max_units, QmpSlot* slots, unsigned long long* generation,
                                                   cudaStream_t stream, QmpMemo* memo) {
    QmpInlineDescs inl;
    for (int i = 0; i < kQmpInlineDescs; ++i) inl.d[i] = descs_host[i < count ? i : 0];
    const int test_withhold_slot = g_test_break_waits;
    const unsigned long long nonce = qmp_next_nonce();
    // every CTA must be resident at once (they exchange partial sums): never more CTAs than this
    // device has SMs, and never more than the workspace has slots
    const unsigned cap = static_cast<unsigned>(std::min(device_sm_count(), kQmpMaxCtas));
    const unsigned grid = max_units < cap ? max_units : cap;
    if (!ensure_dynamic_smem<quantize_mask_pack_stream_kernel<PATTERN, SINGLE>>(kQmpStreamSmemBytes)) return SBN_ERR_CUDA;
    // At most one CTA per SM (kQmpThreads threads of up to 80 registers; kQmpStreamSmemBytes and a few KB more of shared memory) and
    // never more CTAs than SMs, so all of them become resident as soon as the SMs are free and the exchange cannot deadlock; if
    // another kernel kept SMs busy for seconds, the bounded wait reports SBN_ERR_TIMEOUT instead.
    const cudaError_t err = launch_kernel(quantize_mask_pack_stream_kernel<PATTERN, SINGLE>, dim3(grid), dim3(kQmpThreads), kQmpStreamSmemBytes, stream,
                                          inl, rest_dev, count, slots, generation, nonce, test_withhold_slot, count == 1 ? memo : nullptr, qmp_magic(grid));
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}
template <int PATTERN>
inline sbn_status launch_quantize_mask_pack_stream(const QmpDesc* descs_host, const QmpDesc* rest_dev, int count,
                                                   uint32_t max_units, QmpSlot* slots, unsigned long long* generation,
                                                   cudaStream_t stream, QmpMemo* memo = nullptr) {
    if (count == 1) return launch_quantize_mask_pack_stream_cfg<PATTERN, true>(descs_host, rest_dev, count, max_units, slots, generation, stream, memo);
    if constexpr (PATTERN == 24) return launch_quantize_mask_pack_stream_cfg<24, false>(descs_host, rest_dev, count, max_units, slots, generation, stream, memo);
    return SBN_ERR_UNSUPPORTED;                              // no batches of 6:8
}

template <int PATTERN>
inline sbn_status launch_quantize_mask_pack(const void* W, bool w_bf16, int N, int K, int8_t* vals,
                                            uint8_t* meta, float* w_scale, int8_t* dense_q,
                                            const uint8_t* prev_meta,
                                            unsigned long long* flip_bits, QmpWorkspace* ws,
                                            cudaStream_t stream) {
    const QmpDesc d = qmp_make_desc(W, w_bf16, N, K, vals, meta, w_scale, dense_q, prev_meta, flip_bits);
    // the scale a call leaves behind is for the next 2:4 call only; 6:8 always samples (its tag names neither pattern nor dtype)
    return launch_quantize_mask_pack_stream<PATTERN>(&d, nullptr, 1, d.num_units, ws->slot, &ws->generation, stream,
                                                     PATTERN == 24 ? &ws->memo : nullptr);
}

}  // namespace sbn
