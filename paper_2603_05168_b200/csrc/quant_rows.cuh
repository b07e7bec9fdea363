// The activation quantisers (quant_act.cuh, norm_quant_act.cuh) for many rows: a warp per row, rows through shared memory.
//
// With several warps per row the instructions of those kernels go into what every thread does once per row -- reductions,
// two barriers, a square root and three divisions, about 200 instructions for 20 elements of a thread -- and
// the next row's registers.  Here a warp owns a row: the per-row work is spread over K / 32 elements of a lane, nothing is shared
// between warps, and a row arrives by a bulk copy into the warp's own piece of shared memory, which costs neither registers nor
// issue slots.  Up to 32 warps, as many rows as fit in flight.  The row is read from shared memory once per step (squares, maximum,
// codes); xn is computed again rather than kept.
//
// Measured in a chain of launches, us, those kernels / this one [HBM time of the bytes]: plain 4096 x 2560 7.7 / 7.2 [4.9], 4096 x
// 3328 10.8 / 8.9 [6.3], 8192 x 4096 22.5 / 19.5 [15.6]; with norm and gain 2048 x 2560 8.2 / 6.8, 4096 x 2560 12.3 / 11.4, 8192 x
// 2560 22.1 / 19.5 [9.7].  The norm is bound by its instructions (18 per element, before 26).  Two rows per warp (twice the
// independent work, gains read once for both) were slower, two stages per warp too (half the warps).
#pragma once

#include "gemm_tcgen05.cuh"
#include "norm_quant_act.cuh"

namespace sbn {

constexpr int kRowsMaxWarps = 32;
constexpr int kRowsSmemBytes = 200 * 1024;
// Never two CTAs on an SM: the ones that come early, while the kernel before still runs, crowd on the SMs that it has left and
// the others stay idle (norm of 2048 x 2560 8.3 us, with one CTA per SM 6.9).
constexpr int kRowsSmemLeast = 116 * 1024;

__device__ __forceinline__ uint4 lds_vec(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// Scale and codes of a plain row with a NaN (lying at `at` in shared memory): the maximum part by part (see row_parts).  Stored over the
// ones before by a call that is hardly ever made; code for it at the maximum cost every call 2 to 4 % (4096 x 1024 3.26 / 3.38 us).
__device__ __noinline__ void nan_row_codes(uint32_t at, int row, int nvec, uint32_t lane, uint2* xq, size_t tb8, float* a_scale) {
    const int parts = row_parts(nvec);
    float amax = 0.0f;
#pragma unroll 1
    for (int p = 0; p < parts; ++p) {
        uint32_t pm = 0u;
#pragma unroll 1
        for (int idx = 32 * p + lane; idx < nvec; idx += 32 * parts) pm = absmax8_packed(lds_vec(at + 16u * idx), pm);
        amax = fmaxf(amax, __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, max(pm >> 16, pm & 0xFFFFu)) << 16));
    }
    const float d = fmaxf(amax, kEps);
    const float s_x = __fdiv_rn(127.0f, d);
    if (lane == 0u) a_scale[row] = __fdiv_rn(d, 127.0f);
#pragma unroll 1
    for (int idx = lane; idx < nvec; idx += 32) {
        const uint4 v = lds_vec(at + 16u * idx);
        store_codes8<false>(xq, row, idx, tb8, make_uint2(quant_pair2(v.x, v.y, s_x), quant_pair2(v.z, v.w, s_x)));
    }
}

// Shared memory: gains [2][nvec] float4 (first halves of all vectors, then the second ones) when GAIN, then a row per warp.
template <bool NORM, bool GAIN>
__global__ void __launch_bounds__(32 * kRowsMaxWarps, 1)
quant_rows_kernel(const uint4* __restrict__ x, int T, int nvec, const float4* __restrict__ gain, float eps, double n, double inv_n,
                  uint2* __restrict__ xq, float* __restrict__ a_scale) {
    extern __shared__ __align__(128) uint8_t s_rows[];
    __shared__ unsigned long long s_bar[kRowsMaxWarps];
    __shared__ int s_abort;
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t row_bytes = static_cast<uint32_t>(nvec) * 16u;
    const float4* const s_gain = reinterpret_cast<const float4*>(s_rows);
    const uint32_t at = smem_u32(s_rows) + (GAIN ? 2u * row_bytes : 0u) + static_cast<uint32_t>(warp) * row_bytes;
    const uint32_t bar = smem_u32(&s_bar[warp]);
    const size_t tb8 = xq_tb8(T);
    const int stride = gridDim.x * warps;
    int row = blockIdx.x * warps + warp;

    pdl_launch_dependents();
    if (threadIdx.x == 0) s_abort = 0;
    if (lane == 0u) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (lane == 0u && row < T) prefetch_l2_bulk(x + static_cast<size_t>(row) * nvec, row_bytes);       // see quant_act.cuh
    if constexpr (GAIN) {
        for (int i = threadIdx.x; i * 4 < nvec; i += blockDim.x) prefetch_l2_line(gain + 8 * i);
    }
    pdl_wait();
    auto fetch = [&](int r) {
        if (lane == 0u && r < T) {
            mbar_expect_tx(bar, row_bytes);
            bulk_load_once(at, x + static_cast<size_t>(r) * nvec, row_bytes, bar, l2_policy_evict_first());
        }
    };
    fetch(row);
    if constexpr (GAIN) {
        for (int i = threadIdx.x; i < nvec; i += blockDim.x) {
            reinterpret_cast<float4*>(s_rows)[i] = __ldg(gain + 2 * i);
            reinterpret_cast<float4*>(s_rows)[nvec + i] = __ldg(gain + 2 * i + 1);
        }
    }
    __syncthreads();
    for (uint32_t parity = 0u; row < T; parity ^= 1u, row += stride) {
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, &s_abort))) {
            int keep_waiting = 0;                                               // the copy in flight must land before this CTA leaves
            mbar_wait(bar, parity, &keep_waiting);
            break;
        }
        float rinv = 1.0f, amax;
        auto normalise = [&](const uint4& v, int idx, uint64_t (&o)[4]) {
            normalise8(v, pack_f32x2(rinv, rinv), o);
            if constexpr (GAIN) apply_gain8(s_gain[idx], s_gain[nvec + idx], o);
        };
        if constexpr (NORM) {
            double s4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
            for (int idx = lane; idx < nvec; idx += 32) add_squares8(lds_vec(at + 16u * idx), s4);
            double ss = (s4[0] + s4[1]) + (s4[2] + s4[3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
            rinv = norm_factor(ss, n, inv_n, eps);
            amax = 0.0f;
#pragma unroll 4
            for (int idx = lane; idx < nvec; idx += 32) {
                uint64_t o[4];
                normalise(lds_vec(at + 16u * idx), idx, o);
                amax = max_abs8(o, amax);
            }
            amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax)));
        } else {
            uint32_t pm = 0u;
#pragma unroll 4
            for (int idx = lane; idx < nvec; idx += 32) pm = absmax8_packed(lds_vec(at + 16u * idx), pm);
            amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, max(pm >> 16, pm & 0xFFFFu)) << 16);
        }
        const float d = fmaxf(amax, kEps);
        const float s_x = __fdiv_rn(127.0f, d);
        if (lane == 0u) a_scale[row] = __fdiv_rn(d, 127.0f);
        const uint64_t s2 = pack_f32x2(s_x, s_x);
#pragma unroll 4
        for (int idx = lane; idx < nvec; idx += 32) {
            const uint4 v = lds_vec(at + 16u * idx);
            uint2 ov;
            if constexpr (NORM) {
                uint64_t o[4];
                normalise(v, idx, o);
                ov = round_codes8(o, s2);
            } else {
                ov = make_uint2(quant_pair2(v.x, v.y, s_x), quant_pair2(v.z, v.w, s_x));
            }
            store_codes8<false>(xq, row, idx, tb8, ov);
        }
        if constexpr (NORM) {
            if (fmaxf(d, rinv) == __int_as_float(0x7F800000)) odd_row_codes<32, false>(x, gain, rinv, row, nvec, lane, xq, tb8);
        } else {
            if (__float_as_uint(amax) > 0x7F800000u) nan_row_codes(at, row, nvec, lane, xq, tb8, a_scale);
        }
        __syncwarp();                                                           // every lane has read the row
        fetch(row + stride);
    }
}

template <bool NORM, bool GAIN>
static cudaError_t launch_quant_rows(const void* x, int T, int K, const float* gain, float eps, int8_t* xq, float* a_scale, cudaStream_t stream) {
    auto kernel = quant_rows_kernel<NORM, GAIN>;
    if (!ensure_dynamic_smem<quant_rows_kernel<NORM, GAIN>>(kRowsSmemBytes)) return cudaErrorUnknown;
    const int row_bytes = 2 * K, gain_bytes = GAIN ? 4 * K : 0, sms = device_sm_count();
    const int most = std::min(kRowsMaxWarps, (kRowsSmemBytes - gain_bytes) / row_bytes);
    const int rounds = (T + sms * most - 1) / (sms * most), warps = (T + sms * rounds - 1) / (sms * rounds);     // the last round full
    const int grid = std::min(sms, (T + warps - 1) / warps);
    ++g_launch_count;
    return launch_kernel(kernel, dim3(grid), dim3(32 * warps), static_cast<size_t>(std::max(kRowsSmemLeast, gain_bytes + warps * row_bytes)), stream,
                         static_cast<const uint4*>(x), T, K / 8, reinterpret_cast<const float4*>(gain), eps, static_cast<double>(K), 1.0 / static_cast<double>(K),
                         reinterpret_cast<uint2*>(xq), a_scale);
}

// Which calls run here.  Plain: from 13 rows per SM on (2560 columns, 1500 rows 3.8 us there, 4.0 here; 2048 rows 4.8 / 4.7), up to 5120
// columns (8192 x 5120 26.1 / 24.1; 8192 x 6912 32.3 / 32.6: too few rows in flight).  With a norm earlier, 1280 to 3328 columns
// (1000 x 2560 5.9 / 5.0; narrower rows have no advantage), wider ones only in great numbers (8192 x 4096 30.7 / 27.9, 4096 x 4096 16.7 / 18.8).
// Not the expanded form of the 6:8 pattern (2048 x 2560 6.0 / 6.7).
inline bool quant_rows_takes(bool norm, int T, int K) {
    if (norm) return (K >= 1280 && K <= 3328 && T >= 1000) || (K > 3328 && K <= 5120 && T >= 7000);
    return K >= 1024 && K <= 5120 && T >= 13 * kNumSMs;
}

inline sbn_status quantise(const void* x, int T, int K, int8_t* xq, float* a_scale, cudaStream_t stream) {
    if (!quant_rows_takes(false, T, K)) return launch_quant_act(x, T, K, xq, a_scale, stream);
    return launch_quant_rows<false, false>(x, T, K, nullptr, 0.0f, xq, a_scale, stream) == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}
inline sbn_status normalise_and_quantise(const void* x, int T, int K, const float* gain, float eps, int8_t* xq, float* a_scale, cudaStream_t stream) {
    if (!quant_rows_takes(true, T, K)) return launch_norm_quant_act(x, T, K, gain, eps, xq, a_scale, stream);
    const cudaError_t err = gain ? launch_quant_rows<true, true>(x, T, K, gain, eps, xq, a_scale, stream)
                                 : launch_quant_rows<true, false>(x, T, K, gain, eps, xq, a_scale, stream);
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

}  // namespace sbn
