// Operands of the backward GEMMs (dual straight-through estimator, Sec. 2.3, Eq. 5; Algorithm 2's
// backward) in bf16, as the tensor-core kernel of gemm_bf16_pair_tcgen05.cuh reads them:
//
//   dX[t][k] = sum_n dY[t][n] * w_masked[n][k]   contraction over n: B = W_eff [N][K]
//   dW[n][k] = sum_t dY[t][n] * x_q[t][k]        contraction over t: B = x_q [T][K]
//
// Both are row-major with the contraction down the rows; the MMA reads them MN-major, so nothing is transposed.
// x_q[t][k] = bf16(x~[t][k] * a_scale[t]) are the fake-quantised activations as a bf16 training run holds
// them; W_eff is written as +-1.0 / 0.0 and its scale is applied once in the GEMM's epilogue.
//
// The work is cut into items of 128 threads, memory-bound (2.6 and 3 bytes per element): 8 lanes per row, so that a warp
// reads whole rows of a tile and every lane writes a full 32-byte sector; both operands in one launch.
// 2560 -> 3840 at 4096 tokens 9.7 us (two launches, W_eff transposed through shared memory: 16.6), 2560 -> 6912 11.4 (20.6),
// 6912 -> 2560 21 (31).
#pragma once

#include "sbn_common.cuh"
#include "layouts.cuh"

namespace sbn {

constexpr int kPrepThreads = 128;                              // one item at a time
constexpr int kPrepItemTokens = 64;                            // x_q item: 64 tokens x 128 columns; W_eff item: 128 x 128

struct PrepJob {
    const uint8_t* vals;                                       // W_eff from the compressed 2:4 form (tiled)
    const uint8_t* meta;
    uint16_t* w_out;
    const uint8_t* xq;                                         // x_q from the tiled int8 activations and their scales
    const float* a_scale;
    uint16_t* x_out;
    int T, N, K;
    int w_items, x_items;                                      // 0: not wanted
};

__device__ __forceinline__ void st_global_32b(void* p, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// +-1.0, 0.0 in bf16 from the byte of a ternary value
__device__ __forceinline__ uint32_t ternary_bf16(uint32_t byte) { return (byte & 1u) * 0x3F80u | ((byte & 0x80u) << 8); }

// Item of W_eff: 128 rows x 128 columns, `tid` of 128 threads.
__device__ __forceinline__ void prep_w_item(const PrepJob& j, int item, int tid) {
    const int KB = j.K >> 7;
    const int kb = item % KB, nb = item / KB;
    const uint32_t r0 = static_cast<uint32_t>(tid) >> 3, c = static_cast<uint32_t>(tid) & 7u;     // 8 value bytes = 4 groups = 16 columns
    const uint8_t* vt = j.vals + static_cast<size_t>(item) * 8192;
    const uint8_t* mt = j.meta + static_cast<size_t>(item) * 2048;
    uint16_t* out = j.w_out + (static_cast<size_t>(nb) * 128) * j.K + static_cast<size_t>(kb) * 128 + c * 16;
    uint2 v[8];
    uint32_t m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t r = r0 + 16u * i;
        v[i] = __ldg(reinterpret_cast<const uint2*>(vt + vals_in_tile(r, 8u * c)));
        m[i] = __ldg(reinterpret_cast<const unsigned short*>(mt + r * 16 + c * 2));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        uint32_t o[8];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t pair = (g < 2 ? v[i].x : v[i].y) >> (16 * (g & 1));
            const uint32_t nib = m[i] >> (4 * g);
            const unsigned long long q = (static_cast<unsigned long long>(ternary_bf16(pair & 0xFFu)) << (16 * (nib & 3u))) |
                                         (static_cast<unsigned long long>(ternary_bf16((pair >> 8) & 0xFFu)) << (16 * ((nib >> 2) & 3u)));
            o[2 * g] = static_cast<uint32_t>(q);
            o[2 * g + 1] = static_cast<uint32_t>(q >> 32);
        }
        st_global_32b(out + static_cast<size_t>(r0 + 16u * i) * j.K, o);
    }
}

// Item of x_q: 64 tokens x 128 columns.
__device__ __forceinline__ void prep_x_item(const PrepJob& j, int item, int tid) {
    const int KB = j.K >> 7;
    const int kb = item % KB, t0 = (item / KB) * kPrepItemTokens;
    const int r0 = tid >> 3, c = tid & 7;                      // 16 codes
    const size_t tb8 = xq_tb8(j.T);
    uint4 v[4];
    float s[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = t0 + r0 + 16 * i;
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        s[i] = 0.0f;
        if (t < j.T) {
            v[i] = __ldg(reinterpret_cast<const uint4*>(j.xq + (static_cast<size_t>(kb) * tb8 + (static_cast<uint32_t>(t) >> 3)) * 1024 + (t & 7) * 128 + ((c ^ (t & 7)) << 4)));
            s[i] = __ldg(j.a_scale + t);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = t0 + r0 + 16 * i;
        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        uint32_t o[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const float q0 = static_cast<float>(static_cast<int8_t>((w[p >> 1] >> (16 * (p & 1))) & 0xFFu));
            const float q1 = static_cast<float>(static_cast<int8_t>((w[p >> 1] >> (16 * (p & 1) + 8)) & 0xFFu));
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o[p]) : "f"(__fmul_rn(q1, s[i])), "f"(__fmul_rn(q0, s[i])));
        }
        if (t < j.T) st_global_32b(j.x_out + static_cast<size_t>(t) * j.K + static_cast<size_t>(kb) * 128 + c * 16, o);
    }
}

__global__ void __launch_bounds__(kPrepThreads)
backward_prep_kernel(const PrepJob j) {
    pdl_launch_dependents();
    pdl_wait();
    const int items = j.w_items + j.x_items;
    for (int i = blockIdx.x; i < items; i += gridDim.x) {
        if (i < j.w_items) prep_w_item(j, i, threadIdx.x);
        else prep_x_item(j, i - j.w_items, threadIdx.x);
    }
}

}  // namespace sbn
