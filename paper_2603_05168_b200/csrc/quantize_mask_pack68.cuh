// The 6:8 pattern (Sec. 2.2: of every 8 consecutive input weights the 6 largest |w| are kept; the
// pattern of the paper's main results) on tensor cores that only know 2:4.
//
// Three overlapping 4-column windows cover a group of 8 columns:
//     window 0 = columns 0..3,   window 1 = columns 2..5,   window 2 = columns 4..7.
// Whatever 6 columns a group keeps, they can be dealt out so that every window holds exactly two
// of them (at most two columns are missing, so columns 0..3 keep >= 2 and 4..7 keep >= 2: window 0
// takes what is kept of {0,1} and fills up from {2,3}, window 2 takes what is kept of {6,7} and
// fills up from {4,5}, and exactly two kept columns of {2..5} remain for window 1).  A 6:8 matrix
// [N][K] is therefore a 2:4 matrix [N][K' = 3K/2] over activations whose rows are expanded the
// same way (K' column 12 g + 4 w + s  <-  column 8 g + 2 w + s; see quant_act.cuh), and the
// sparse GEMM runs unchanged at 3/4 of the dense MMA work.  The outputs are the compressed values
// and metadata of that [N][K'] matrix in the tiled layouts of layouts.cuh.
//
// The pack kernel is the 2:4 one (quantize_mask_pack_stream.cuh) with another pass 1: a group's kept set is
// an index into a table (in shared memory) that says which columns the windows take, in which order.
#pragma once

#include "quantize_mask_pack.cuh"

namespace sbn {

// Eq. 2 for one group of 8: bit j set = column j kept.  The two smallest |w| are dropped; among
// equal magnitudes the higher column goes first (the lower column wins a tie, as in the 2:4 rule).
// t2 = the second smallest (a merge network of sorted pairs); what is larger is kept, and unless there is a tie at t2
// that is all of it.
__device__ __forceinline__ uint32_t select6of8(const float (&a)[8]) {
    float lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { lo[i] = fminf(a[2 * i], a[2 * i + 1]); hi[i] = fmaxf(a[2 * i], a[2 * i + 1]); }
    const float l0 = fminf(lo[0], lo[1]), s0 = fmin3(fmaxf(lo[0], lo[1]), hi[0], hi[1]);
    const float l1 = fminf(lo[2], lo[3]), s1 = fmin3(fmaxf(lo[2], lo[3]), hi[2], hi[3]);
    const float t2 = fmin3(fmaxf(l0, l1), s0, s1);
    uint32_t S = qmp_byte_bits(sign_bytes4(t2 - a[0], t2 - a[1], t2 - a[2], t2 - a[3]), sign_bytes4(t2 - a[4], t2 - a[5], t2 - a[6], t2 - a[7]));
    int need = 6 - __popc(S);
    if (need != 0) {                                          // a tie: the lowest of the columns that equal t2
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (need != 0 && a[i] == t2) { S |= 1u << i; --need; }
        }
    }
    return S;
}

// The same for two groups of bf16 weights at once, in halfword arithmetic: r[0 .. 3] and r[4 .. 7] are the groups' words.  Ties
// are common with 8 significant bits, so their path is short too.
__device__ __forceinline__ void select6of8_bf16(const uint32_t (&r)[8], uint32_t& S0, uint32_t& S1) {
    uint32_t p[8];                                            // column j of both groups
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = r[i] & kAbs2, b = r[4 + i] & kAbs2;
        p[2 * i] = prmt(a, b, 0x5410u);
        p[2 * i + 1] = prmt(a, b, 0x7632u);
    }
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { lo[i] = __vminu2(p[2 * i], p[2 * i + 1]); hi[i] = __vmaxu2(p[2 * i], p[2 * i + 1]); }
    const uint32_t l0 = __vminu2(lo[0], lo[1]), s0 = __vminu2(__vmaxu2(lo[0], lo[1]), __vminu2(hi[0], hi[1]));
    const uint32_t l1 = __vminu2(lo[2], lo[3]), s1 = __vminu2(__vmaxu2(lo[2], lo[3]), __vminu2(hi[2], hi[3]));
    const uint32_t t2 = __vminu2(__vmaxu2(l0, l1), __vminu2(s0, s1));
    // flags in bits 15 and 31 of eight words -> a bit per column, group 0 in byte 0, group 1 in byte 1
    auto gather = [](const uint32_t (&f)[8]) {
        const uint32_t y = (prmt(f[0], f[1], kSign2) & 0x02020101u) | (prmt(f[2], f[3], kSign2) & 0x08080404u) |
                           (prmt(f[4], f[5], kSign2) & 0x20201010u) | (prmt(f[6], f[7], kSign2) & 0x80804040u);
        return (y | (y >> 16)) & 0xFFFFu;
    };
    uint32_t f[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) f[j] = sub_abs_bf16x2(t2, p[j]);
    uint32_t drop = gather(f) ^ 0xFFFFu;                      // |w| <= t2: dropped, unless there are more than two
    if (__popc(drop) != 4) {
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = sub_abs_bf16x2(p[j], t2);
        uint32_t less = gather(f), same = drop & ~less;       // the highest of the equal columns go
        uint32_t s_lo = same & 0xFFu, s_hi = same >> 8;
        while (__popc(s_lo) + __popc(less & 0xFFu) > 2) s_lo &= s_lo - 1u;
        while (__popc(s_hi) + __popc(less >> 8) > 2) s_hi &= s_hi - 1u;
        drop = less | s_lo | (s_hi << 8);
    }
    S0 = ~drop & 0xFFu;
    S1 = (~drop >> 8) & 0xFFu;
}

// Deals the kept columns S (6 bits set of 8) out to the three windows: 4-bit masks, two bits each.
__device__ __forceinline__ void windows68(uint32_t S, uint32_t& m0, uint32_t& m1, uint32_t& m2) {
    const uint32_t L = S & 3u, ML = (S >> 2) & 3u, MR = (S >> 4) & 3u, R = (S >> 6) & 3u;
    const uint32_t need_l = 2u - __popc(L);
    const uint32_t take_l = need_l == 0u ? 0u : (need_l == 1u ? (ML & (0u - ML)) : ML);        // lowest first
    const uint32_t need_r = 2u - __popc(R);
    const uint32_t take_r = need_r == 0u ? 0u : (need_r == 1u ? (MR == 3u ? 2u : MR) : MR);    // highest first
    m0 = L | (take_l << 2);
    m2 = take_r | (R << 2);
    m1 = (ML & ~take_l) | ((MR & ~take_r) << 2);
}

// 2:4 metadata nibble (i0 | i1 << 2, i0 < i1) of a 4-bit mask with exactly two bits set.
__device__ __forceinline__ uint32_t mask4_to_nibble(uint32_t m) {
    constexpr uint32_t kLo = (4u << 12) | (8u << 20) | (9u << 24);      // masks 3, 5, 6
    constexpr uint32_t kHi = (12u << 4) | (13u << 8) | (14u << 16);     // masks 9, 10, 12
    return (((m & 8u) ? kHi : kLo) >> (4u * (m & 7u))) & 15u;
}
// Table entry of the kept set S: x = columns of the six kept values, a nibble each, window by window (a byte-permute
// selector for the group's eight value bytes); y = the three windows' metadata nibbles.  Window by window the columns
// ascend (window 0 takes the lowest kept ones, window 2 the highest), so column j is kept value popc(S & (2^j - 1)).
__device__ __forceinline__ uint2 table68_entry(uint32_t S) {
    if (__popc(S) != 6) return make_uint2(0u, 0u);
    uint32_t m[3];
    windows68(S, m[0], m[1], m[2]);
    uint2 e = make_uint2(0u, 0u);
#pragma unroll
    for (uint32_t w = 0; w < 3; ++w) {
        const uint32_t first = __ffs(static_cast<int>(m[w])) - 1, last = 31 - __clz(static_cast<int>(m[w]));
        e.x |= ((2u * w + first) | ((2u * w + last) << 4)) << (8u * w);
        e.y |= mask4_to_nibble(m[w]) << (4u * w);
    }
    return e;
}

// Kept-column mask of a group of 8 from its three metadata nibbles.
__device__ __forceinline__ uint32_t mask8_from_meta12(uint32_t m12) {
    return nibble_to_mask(m12 & 15u) | (nibble_to_mask((m12 >> 4) & 15u) << 2) | (nibble_to_mask((m12 >> 8) & 15u) << 4);
}

// byte offset in the tiled metadata of byte column b of row n (K' space, KBp = K'/128)
__device__ __forceinline__ size_t meta68_offset(uint32_t n, uint32_t b, uint32_t KBp) {
    return (static_cast<size_t>(n >> 7) * KBp + (b >> 4)) * 2048u + ((n & 127u) << 4) + (b & 15u);
}
// byte offset in the tiled values of compressed byte column c of row n
__device__ __forceinline__ size_t vals68_offset(uint32_t n, uint32_t c, uint32_t KBp) {
    return (static_cast<size_t>(n >> 7) * KBp + (c >> 6)) * 8192u + vals_in_tile(n & 127u, c & 63u);
}

// Eq. 1 for the eight weights of a group as bytes (+1 -> 0x01, -1 -> 0xFF, 0 -> 0x00), +-1 iff |w| > thr_pred; `e` =
// the bits of thr_pred - |w|.
__device__ __forceinline__ void ternary68(const float (&w)[8], const float thr_pred, uint32_t (&e)[8], uint32_t& b03, uint32_t& b47) {
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = __float_as_uint(thr_pred - fabsf(w[i]));
    b03 = (sign_bytes4(w[0], w[1], w[2], w[3]) | 0x01010101u) & sign_bytes4(e[0], e[1], e[2], e[3]);
    b47 = (sign_bytes4(w[4], w[5], w[6], w[7]) | 0x01010101u) & sign_bytes4(e[4], e[5], e[6], e[7]);
}

// Values of this CTA's range again with the exact threshold (what qmp_pass2_full is for 2:4): a half-warp per unit, a lane
// one group.
template <bool BF16>
__device__ __forceinline__ void qmp68_pass2_full(const QmpDesc& d, const QmpRange rg, const float thr, const uint2* table) {
    const uint32_t l16 = threadIdx.x & 15u;
    const uint32_t KB = d.KB, KBp = KB + (KB >> 1);           // K' / 128
    const float thr_pred = __uint_as_float(__float_as_uint(thr) - 1u);
    uint8_t* const vals = reinterpret_cast<uint8_t*>(d.vals);
    for (uint32_t u = rg.u_begin + (threadIdx.x >> 4); u < rg.u_end; u += 2u * kQmpWarps) {
        const uint32_t n = u / KB, kb = u - n * KB;
        float4 va, vb;
        qmp_load_group_pair<BF16>(d.W, u, l16, va, vb);
        const float w[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
        float a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = fabsf(w[i]);
        uint32_t e[8], b03, b47;
        ternary68(w, thr_pred, e, b03, b47);
        const uint32_t sel = table[select6of8(a)].x;
        const uint32_t v4 = prmt(b03, b47, sel & 0xFFFFu), v2 = prmt(b03, b47, sel >> 16);
        const uint32_t c = 96u * kb + 6u * l16;
        *reinterpret_cast<uint16_t*>(vals + vals68_offset(n, c, KBp)) = static_cast<uint16_t>(v4);
        *reinterpret_cast<uint16_t*>(vals + vals68_offset(n, c + 2u, KBp)) = static_cast<uint16_t>(v4 >> 16);
        *reinterpret_cast<uint16_t*>(vals + vals68_offset(n, c + 4u, KBp)) = static_cast<uint16_t>(v2);
    }
}

}  // namespace sbn
