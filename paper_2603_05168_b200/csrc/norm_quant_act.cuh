// x~ = Q_a(Norm(x)) (Algorithm 1, forward), Norm read as RMSNorm with a per-channel gain g:
//
//   ms = mean_k x^2 (fp64 accumulation, one cast to fp32),  r = 1 / sqrt(ms + eps),
//   xn = (x * r) * g,   then Q_a of Sec. 2.1 on the fp32 xn:
//   a = max_k |xn|, d = max(a, 1e-5), s_x = 127 / d, xq = clamp(rint(xn * s_x), -128, 127), a_scale = d / 127
//
// One kernel, x read once: the row stays in registers (as bf16) through the three steps -- sum of
// squares, maximum of |xn|, rounding -- and xn is recomputed (two multiplies) instead of stored.
// HBM-bound like the plain quantiser: 2 B read + 1 B written per element; the normalised
// activations never exist in memory.  Same persistent-CTA row pipeline and the same tiled xq
// layout as quant_act.cuh.  The squares of bf16 values are added in fp64 in a fixed order (thread-local, then a
// butterfly, then the warps in order).
//
// Measured in a chain of launches, with a gain (us; HBM time of the bytes in brackets): 1 x 2560 1.57, 16 x 4096 1.8,
// 201 x 2560 2.5 -- two trips to memory, two barriers and the arithmetic between them; 4096 x 2560 11.8 [4.9],
// 4096 x 6912 26.8 [13.2], 8192 x 4096 29.7 [15.6], 8192 x 11008 76 [42] -- bound by the instructions, 22.7 per element
// (73 % of the issue slots busy); the plain quantiser (7.4, 16.3, 21.8, 49) needs fewer.  Squares through the conversion instruction, gains
// fetched before the row, a division for the mean and a clamp: 2.21, 2.10, 3.14, 12.0, 28.2, 31.6 and 82.  One or two
// warps per row without the prefetch of the next row were slower: 15.7, 31.7, 36.6, 90.  Many rows of up to 5120 columns go to
// quant_rows.cuh.
#pragma once

#include "quant_act.cuh"

namespace sbn {

// packed fp32x2 arithmetic (two IEEE round-to-nearest operations per instruction)
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// max(m, |a|, |b|) in one instruction
__device__ __forceinline__ float max_abs3(float m, float a, float b) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(m), "f"(a), "f"(b));
    return d;
}
// The low bytes of four words, lowest first.
__device__ __forceinline__ uint32_t low_bytes4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}
// |value| of a finite bf16 (its 15 bits) as a double: the exponent moves to the double's bias, the significand to the
// top of the high word -- two integer instructions; the conversion instruction runs at an eighth of their rate.  Zero and
// subnormals come out as up to 2^-126 instead; their squares (below 2^-251 each) vanish in the mean's cast to fp32
// (smallest value 2^-149) either way.
__device__ __forceinline__ double bf16_abs_to_f64(uint32_t abs15) {
    return __hiloint2double(static_cast<int>((abs15 << 13) + 0x38000000u), 0);
}

// The arithmetic that every form of the kernel shares, 8 columns (a vector) at a time.
// Adds the squares in fp64, four chains so that the adds overlap: exact products, one rounding in the add.
__device__ __forceinline__ void add_squares8(const uint4& v, double (&s4)[4]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double lo = bf16_abs_to_f64(w[j] & 0x7FFFu), hi = bf16_abs_to_f64((w[j] >> 16) & 0x7FFFu);
        s4[(2 * j) & 3] = __fma_rn(lo, lo, s4[(2 * j) & 3]);
        s4[(2 * j + 1) & 3] = __fma_rn(hi, hi, s4[(2 * j + 1) & 3]);
    }
}
// r from the sum of squares.  ss / n, correctly rounded, from the rounded reciprocal: quotient, exact remainder, correction
// (Markstein's theorem for division with a correctly rounded reciprocal).
__device__ __forceinline__ float norm_factor(double ss, double n, double inv_n, float eps) {
    const double quot = ss * inv_n;
    const float ms = static_cast<float>(__fma_rn(__fma_rn(-quot, n, ss), inv_n, quot));
    return __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(ms, eps)));
}
// xn = (x * r) * g with packed fp32x2 multiplies: both factors of all pairs, then the gains.
__device__ __forceinline__ void normalise8(const uint4& v, uint64_t r2, uint64_t (&out)[4]) {
    out[0] = mul_f32x2(pack_f32x2(bf16lo_to_f32(v.x), bf16hi_to_f32(v.x)), r2);
    out[1] = mul_f32x2(pack_f32x2(bf16lo_to_f32(v.y), bf16hi_to_f32(v.y)), r2);
    out[2] = mul_f32x2(pack_f32x2(bf16lo_to_f32(v.z), bf16hi_to_f32(v.z)), r2);
    out[3] = mul_f32x2(pack_f32x2(bf16lo_to_f32(v.w), bf16hi_to_f32(v.w)), r2);
}
__device__ __forceinline__ void apply_gain8(const float4& a, const float4& b, uint64_t (&out)[4]) {
    out[0] = mul_f32x2(out[0], pack_f32x2(a.x, a.y));
    out[1] = mul_f32x2(out[1], pack_f32x2(a.z, a.w));
    out[2] = mul_f32x2(out[2], pack_f32x2(b.x, b.y));
    out[3] = mul_f32x2(out[3], pack_f32x2(b.z, b.w));
}
__device__ __forceinline__ float max_abs8(const uint64_t (&xn)[4], float m) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float lo, hi;
        unpack_f32x2(xn[j], lo, hi);
        m = max_abs3(m, lo, hi);
    }
    return m;
}
// rint(xn * s_x): multiply, then add 1.5 * 2^23 -- the adder's round-to-nearest-even IS the rounding of the method, and the
// integer is left in the low mantissa bits.  The adds are scalar: a packed multiply followed by a packed add came out with ONE
// rounding (a fused multiply-add), which breaks exact ties such as 63.5.  The method's clamp cannot act: |xn| <= d (finite), so
// |xn * s_x| <= 127 (1 + 2^-23) and rounds to at most 127.  The code is the low byte; the lowest column is the lowest byte of .x.
__device__ __forceinline__ uint2 round_codes8(const uint64_t (&xn)[4], uint64_t s2) {
    uint32_t q[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float lo, hi;
        unpack_f32x2(mul_f32x2(xn[j], s2), lo, hi);
        q[2 * j] = __float_as_uint(__fadd_rn(lo, 12582912.0f));
        q[2 * j + 1] = __float_as_uint(__fadd_rn(hi, 12582912.0f));
    }
    return make_uint2(low_bytes4(q[0], q[1], q[2], q[3]), low_bytes4(q[4], q[5], q[6], q[7]));
}

// Codes of a finite row whose xn is not finite: mean square 0 with eps = 0 (rinv infinite), or a gain that takes xn out of range
// (s_x = 0).  The product is NaN where xn is infinite or NaN: code 127, as a saturating conversion gives; else 0.  The row is read
// again and its codes stored over the ones before: a call that is never made, 1 % of the kernel's time on average (5 % for 8192 rows
// of 4096; code for it inside the loop 2 to 4 % on average, a minimum per code 3 to 8 %).
template <int G, bool EXPAND68>
__device__ __noinline__ void odd_row_codes(const uint4* x, const float4* gain, float rinv, int row, int nvec, int g, uint2* xq, size_t tb8) {
#pragma unroll 1
    for (int idx = g; idx < nvec; idx += G) {
        const uint4 v = __ldg(x + static_cast<size_t>(row) * nvec + idx);
        uint32_t code[2];
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const uint32_t w0 = h ? v.z : v.x, w1 = h ? v.w : v.y;
            const float4 gn = gain != nullptr ? __ldg(gain + 2 * idx + h) : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
            const float xn[4] = {bf16lo_to_f32(w0) * rinv * gn.x, bf16hi_to_f32(w0) * rinv * gn.y, bf16lo_to_f32(w1) * rinv * gn.z, bf16hi_to_f32(w1) * rinv * gn.w};
            uint32_t c = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) c |= fabsf(xn[j]) < __int_as_float(0x7F800000) ? 0u : 0x7Fu << (8 * j);
            if (h) code[1] = c; else code[0] = c;
        }
        store_codes8<EXPAND68>(xq, row, idx, tb8, make_uint2(code[0], code[1]));
    }
}

// G threads per token row, VPT 16-byte vectors per thread (G * VPT >= K / 8).  GAIN: known at compile time -- with a test of the
// pointer the registers for gains that are not there and a branch per vector cost rows without a gain 4 to 6 % (8192 x 4096 29.1 us,
// now 26.3).
template <int G, int VPT, bool EXPAND68, bool GAIN>
__global__ void __launch_bounds__(kActThreads, (VPT <= 4) ? 3 : 2)
norm_quant_act_kernel(const uint4* __restrict__ x, int T, int nvec, const float4* __restrict__ gain, float eps, double n, double inv_n,
                      uint2* __restrict__ xq, float* __restrict__ a_scale) {
    constexpr int ROWS = kActThreads / G;
    constexpr int WARPS_PER_ROW = (G + 31) / 32;
    __shared__ double s_sum[2][kActThreads / 32];
    __shared__ float s_max[2][kActThreads / 32];

    const int r = threadIdx.x / G;
    const int g = threadIdx.x % G;
    const int warp = threadIdx.x >> 5;
    const int w0 = (r * G) >> 5;                                  // first warp of this row group
    const int row_stride = gridDim.x * ROWS;
    const size_t tb8 = xq_tb8(T);
    const int iters = (T + row_stride - 1) / row_stride;        // same for every thread of the CTA

    pdl_launch_dependents();             // the next kernel may become resident (and fetch weights) right away
    uint4 cur[VPT], nxt[VPT];
    int row = blockIdx.x * ROWS + r;
    // The first row goes to the L2 while the kernel before finishes (see quant_act.cuh).  Not the gains, which are there as a rule: with them
    // rows in the L2 took up to 20 % longer (777 x 4096 4.3 / 5.1 us, 400 x 4096 2.6 / 3.1; from memory 14 % less than without any, 9 % with them).
    if (row < T && g * 8 < nvec) prefetch_l2_line(x + static_cast<size_t>(row) * nvec + g * 8);
    pdl_wait();

    // the first row is on its way before the gains are fetched (one after the other they were two trips to memory)
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int idx = g + i * G;
        cur[i] = (row < T && idx < nvec) ? __ldg(x + static_cast<size_t>(row) * nvec + idx) : make_uint4(0u, 0u, 0u, 0u);
    }
    // The gains of a thread's columns: in registers up to two vectors, else in shared memory -- the first halves of all
    // vectors, then the second ones (one after the other the lanes' reads had two-way bank conflicts).
    constexpr bool GAIN_REGS = VPT <= 2;
    extern __shared__ float4 s_gain[];                           // [2][nvec] when a gain is given
    float4 gain_r[GAIN_REGS ? VPT : 1][2];
    if constexpr (GAIN_REGS) {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int idx = g + i * G;
            gain_r[i][0] = gain_r[i][1] = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
            if (GAIN && idx < nvec) { gain_r[i][0] = __ldg(gain + 2 * idx); gain_r[i][1] = __ldg(gain + 2 * idx + 1); }
        }
    } else if (GAIN) {
        for (int i = threadIdx.x; i < nvec; i += kActThreads) {
            s_gain[i] = __ldg(gain + 2 * i);
            s_gain[nvec + i] = __ldg(gain + 2 * i + 1);
        }
        __syncthreads();
    }
    for (int it = 0; it < iters; ++it, row += row_stride) {
        const int row_n = row + row_stride;
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int idx = g + i * G;
            nxt[i] = (row_n < T && idx < nvec) ? __ldg(x + static_cast<size_t>(row_n) * nvec + idx) : make_uint4(0u, 0u, 0u, 0u);
        }
        // ---- mean square
        double s4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < VPT; ++i) add_squares8(cur[i], s4);
        double ss = (s4[0] + s4[1]) + (s4[2] + s4[3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, o);
        if constexpr (WARPS_PER_ROW > 1) {
            double* sm = s_sum[it & 1];
            if ((threadIdx.x & 31) == 0) sm[warp] = ss;
            __syncthreads();
            double t = 0.0;
#pragma unroll
            for (int w = 0; w < WARPS_PER_ROW; ++w) t += sm[w0 + w];
            ss = t;
        }
        const float rinv = norm_factor(ss, n, inv_n, eps);
        // ---- xn and max |xn|.  Up to four vectors per thread the fp32 xn stays in registers for the rounding; longer rows recompute it.
        constexpr bool KEEP = VPT <= 4;
        const uint64_t r2 = pack_f32x2(rinv, rinv);
        uint64_t xn2[KEEP ? VPT : 1][4];
        float amax = 0.0f;
        auto normalise = [&](const uint4& v, int i, uint64_t (&out)[4]) {
            const int idx = g + i * G;
            normalise8(v, r2, out);
            if (GAIN && idx < nvec) {
                const float4 a = GAIN_REGS ? gain_r[GAIN_REGS ? i : 0][0] : s_gain[idx], b = GAIN_REGS ? gain_r[GAIN_REGS ? i : 0][1] : s_gain[nvec + idx];
                apply_gain8(a, b, out);
            }
        };
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            uint64_t tmp[4];
            uint64_t (&o)[4] = KEEP ? xn2[KEEP ? i : 0] : tmp;
            normalise(cur[i], i, o);
            amax = max_abs8(o, amax);
        }
        // bit patterns of non-negative floats order like integers: one redux instruction per warp
        amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax)));
        if constexpr (WARPS_PER_ROW > 1) {
            float* sm = s_max[it & 1];
            if ((threadIdx.x & 31) == 0) sm[warp] = amax;
            __syncthreads();
            float m = sm[w0];
#pragma unroll
            for (int w = 1; w < WARPS_PER_ROW; ++w) m = fmaxf(m, sm[w0 + w]);
            amax = m;
        }
        if (row < T) {
            const float d = fmaxf(amax, kEps);
            const float s_x = __fdiv_rn(127.0f, d);
            if (g == 0) a_scale[row] = __fdiv_rn(d, 127.0f);
            const uint64_t s2 = pack_f32x2(s_x, s_x);
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const int idx = g + i * G;
                if (idx < nvec) {
                    uint64_t tmp[4];
                    if constexpr (!KEEP) normalise(cur[i], i, tmp);
                    const uint64_t (&o)[4] = KEEP ? xn2[KEEP ? i : 0] : tmp;
                    store_codes8<EXPAND68>(xq, row, idx, tb8, round_codes8(o, s2));     // plain, or expanded for the 6:8 pattern
                }
            }
            if (fmaxf(d, rinv) == __int_as_float(0x7F800000))              // for the whole group of threads, so for whole warps
                odd_row_codes<G, EXPAND68>(x, gain, rinv, row, nvec, g, xq, tb8);
        }
#pragma unroll
        for (int i = 0; i < VPT; ++i) cur[i] = nxt[i];
    }
}

template <int G, int VPT, bool EXPAND68>
static cudaError_t launch_norm_quant_act_cfg(const uint4* x, int T, int nvec, const float4* gain, float eps, uint2* q,
                                             float* a_scale, cudaStream_t stream) {
    constexpr int rows = kActThreads / G;
    const int ctas_per_sm = (VPT <= 4) ? 3 : 2;
    int grid = (T + rows - 1) / rows;
    if (grid > kNumSMs * ctas_per_sm) grid = kNumSMs * ctas_per_sm;
    const size_t smem = gain && VPT > 2 ? static_cast<size_t>(nvec) * 32 : 0;   // K floats
    if (!ensure_dynamic_smem<norm_quant_act_kernel<G, VPT, EXPAND68, true>>(65536)) return cudaErrorUnknown;
    return launch_kernel(gain ? norm_quant_act_kernel<G, VPT, EXPAND68, true> : norm_quant_act_kernel<G, VPT, EXPAND68, false>,
                         dim3(grid), dim3(kActThreads), smem, stream, x, T, nvec, gain, eps, static_cast<double>(nvec * 8), 1.0 / static_cast<double>(nvec * 8), q, a_scale);
}

// K up to 16384 (the register-resident row); longer rows are refused by the caller.
template <bool EXPAND68 = false>
inline sbn_status launch_norm_quant_act(const void* x_bf16, int T, int K, const float* gain, float eps, int8_t* xq,
                                        float* a_scale, cudaStream_t stream) {
    const int nvec = K / 8;
    const uint4* x = static_cast<const uint4*>(x_bf16);
    const float4* g4 = reinterpret_cast<const float4*>(gain);
    uint2* q = reinterpret_cast<uint2*>(xq);
    cudaError_t err;
    // Few rows: one per CTA with all its threads, so that what a thread does between the barriers is short.  With 2560 columns
    // (us, a whole CTA / two rows per CTA): 1.59 / 2.11 at 16 rows, 2.08 / 2.33 at 222, 2.86 / 3.28 at 444 (every row
    // resident), 4.17 / 4.12 at 777; narrower rows cross earlier (1280 columns: 1.59 / 1.80 at 148, 1.85 / 1.78 at 222).
    // Many rows: smaller groups, whose barriers are shared by fewer warps.
    if (T <= kNumSMs * (nvec > 256 ? 3 : 1) && nvec > 128 && nvec <= 256 * 2) err = launch_norm_quant_act_cfg<256, 2, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 32 * 2) err = launch_norm_quant_act_cfg<32, 2, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 64 * 2) err = launch_norm_quant_act_cfg<64, 2, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 128 * 2) err = launch_norm_quant_act_cfg<128, 2, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 128 * 3) err = launch_norm_quant_act_cfg<128, 3, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 256 * 2) err = launch_norm_quant_act_cfg<256, 2, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 256 * 3) err = launch_norm_quant_act_cfg<256, 3, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 256 * 4) err = launch_norm_quant_act_cfg<256, 4, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 256 * 6) err = launch_norm_quant_act_cfg<256, 6, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else if (nvec <= 256 * 8) err = launch_norm_quant_act_cfg<256, 8, EXPAND68>(x, T, nvec, g4, eps, q, a_scale, stream);
    else return SBN_ERR_UNSUPPORTED;
    ++g_launch_count;
    return err == cudaSuccess ? SBN_OK : SBN_ERR_CUDA;
}

}  // namespace sbn
