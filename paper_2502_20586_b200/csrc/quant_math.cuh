// Per-element arithmetic of the quantiser: Philox4x32-10, the sign vector, the in-register Hadamard
// butterflies, the E8M0 scale rule and the E2M1 encoders (Algorithms 1 and 2).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mx {

// ---------------------------------------------------------------- Philox4x32-10 (counter-based)
// key = (seed lo, seed hi); counter = (index lo, index hi, stream_tag, domain).
// domain 0: sign vector (stream_tag 0, index = j / 128).  domain 1: SR draws (index = element / 16).
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint32_t u4_word(const uint4& v, int i) {
    return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// The 32 sign bits of elements [32 w, 32 w + 32) of the g-long sign vector (bit set = -1).
__device__ __forceinline__ uint32_t sign_word(uint64_t seed, int w) {
    const uint4 o = philox4x32_10((uint32_t)(w >> 2), 0u, 0u, 0u, (uint32_t)seed, (uint32_t)(seed >> 32));
    return u4_word(o, w & 3);
}

// The 32 8-bit SR draws of elements [i0, i0 + 32), i0 a multiple of 32: two Philox calls, eight words.
__device__ __forceinline__ void sr_draws32(uint64_t seed, uint32_t stream_tag, uint64_t i0, uint32_t (&rw)[8]) {
    const uint64_t idx = i0 >> 4;
    const uint4 a = philox4x32_10((uint32_t)idx, (uint32_t)(idx >> 32), stream_tag, 1u, (uint32_t)seed, (uint32_t)(seed >> 32));
    const uint4 b = philox4x32_10((uint32_t)(idx + 1), (uint32_t)((idx + 1) >> 32), stream_tag, 1u, (uint32_t)seed, (uint32_t)(seed >> 32));
    rw[0] = a.x; rw[1] = a.y; rw[2] = a.z; rw[3] = a.w;
    rw[4] = b.x; rw[5] = b.y; rw[6] = b.z; rw[7] = b.w;
}

// Same draws with the ten round keys given (they depend on the seed only and come with the kernel's parameters).
struct PhiloxKeys {
    uint32_t k0[10], k1[10];
};
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKeys& ks) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ ks.k0[i];
        c1 = lo1;
        c2 = hi0 ^ c3 ^ ks.k1[i];
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}
// i0 is a multiple of 32, so the two call indices i0/16 and i0/16 + 1 differ in the lowest bit only.
__device__ __forceinline__ void sr_draws32(const PhiloxKeys& ks, uint32_t stream_tag, uint64_t i0, uint32_t (&rw)[8]) {
    const uint32_t lo = (uint32_t)(i0 >> 4), hi = (uint32_t)(i0 >> 36);
    const uint4 a = philox4x32_10(lo, hi, stream_tag, 1u, ks);
    const uint4 b = philox4x32_10(lo | 1u, hi, stream_tag, 1u, ks);
    rw[0] = a.x; rw[1] = a.y; rw[2] = a.z; rw[3] = a.w;
    rw[4] = b.x; rw[5] = b.y; rw[6] = b.z; rw[7] = b.w;
}
// The same for MX block `blk` = i0 / 32 of an operand below 2^36 elements.
__device__ __forceinline__ void sr_draws32_block(const PhiloxKeys& ks, uint32_t stream_tag, uint32_t blk, uint32_t (&rw)[8]) {
    const uint4 a = philox4x32_10(2u * blk, 0u, stream_tag, 1u, ks);
    const uint4 b = philox4x32_10(2u * blk | 1u, 0u, stream_tag, 1u, ks);
    rw[0] = a.x; rw[1] = a.y; rw[2] = a.z; rw[3] = a.w;
    rw[4] = b.x; rw[5] = b.y; rw[6] = b.z; rw[7] = b.w;
}

// The SR draws of one operand view share seed and stream tag, and for operands below 2^36 elements the high counter
// word is zero: the counter is (index, 0, tag, 1).  Everything in the first three rounds that does not depend on the
// index is folded into five words per view (computed on the host with the key schedule): the rounds themselves, and so
// the draws, are unchanged.
struct PhiloxViewConsts {
    uint32_t c1, d, e, f, qlo;
};
__host__ __device__ inline PhiloxViewConsts philox_view_consts(const PhiloxKeys& ks, uint32_t stream_tag) {
    const unsigned long long p1 = 0xCD9E8D57ull * stream_tag;             // round 1: second product, counter word 2 = tag
    const uint32_t a = (uint32_t)(p1 >> 32) ^ 0u ^ ks.k0[0], b = (uint32_t)p1;   // new words 0, 1 (counter word 1 = 0)
    const unsigned long long q = 0xD2511F53ull * a;                       // round 2: first product
    PhiloxViewConsts v;
    v.c1 = 1u ^ ks.k1[0];                                                 // round 1, word 2: hi(M0 x0) ^ (domain 1) ^ key
    v.d = b ^ ks.k0[1];                                                   // round 2, word 0: hi(M1 y2) ^ b ^ key
    v.e = (uint32_t)(q >> 32) ^ ks.k1[1];                                 // round 2, word 2: y3 ^ hi(M0 a) ^ key
    v.qlo = (uint32_t)q;                                                  // round 2, word 3
    v.f = v.qlo ^ ks.k1[2];                                               // round 3, word 2: hi(M0 z0) ^ qlo ^ key
    return v;
}
__device__ __forceinline__ uint4 philox4x32_10_view(uint32_t x0, const PhiloxViewConsts& v, const PhiloxKeys& ks) {
    const uint32_t y2 = __umulhi(0xD2511F53u, x0) ^ v.c1, y3 = 0xD2511F53u * x0;                 // round 1
    const uint32_t z0 = __umulhi(0xCD9E8D57u, y2) ^ v.d, z1 = 0xCD9E8D57u * y2, z2 = y3 ^ v.e;   // round 2
    uint32_t c0 = __umulhi(0xCD9E8D57u, z2) ^ z1 ^ ks.k0[2], c1 = 0xCD9E8D57u * z2;              // round 3
    uint32_t c2 = __umulhi(0xD2511F53u, z0) ^ v.f, c3 = 0xD2511F53u * z0;
#pragma unroll
    for (int i = 3; i < 10; ++i) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ ks.k0[i];
        c1 = lo1;
        c2 = hi0 ^ c3 ^ ks.k1[i];
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}
__device__ __forceinline__ void sr_draws32_view(const PhiloxKeys& ks, const PhiloxViewConsts& v, uint32_t blk, uint32_t (&rw)[8]) {
    const uint4 a = philox4x32_10_view(2u * blk, v, ks);
    const uint4 b = philox4x32_10_view(2u * blk | 1u, v, ks);
    rw[0] = a.x; rw[1] = a.y; rw[2] = a.z; rw[3] = a.w;
    rw[4] = b.x; rw[5] = b.y; rw[6] = b.z; rw[7] = b.w;
}

// ---------------------------------------------------------------- Hadamard butterflies (Eq. 4)
// In-place Sylvester transform over the 32 values of one thread (natural order, un-normalised).
__device__ __forceinline__ void fwht32(float (&v)[32]) {
#pragma unroll
    for (int h = 1; h < 32; h <<= 1) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            if ((i & h) == 0) {
                const float a = v[i], b = v[i + h];
                v[i] = a + b;
                v[i + h] = a - b;
            }
        }
    }
}
// One butterfly stage across lanes that differ in `lane_mask` (lane bit clear holds the "upper" half).
__device__ __forceinline__ void fwht_cross(float (&v)[32], int lane_mask, int lane) {
    const bool upper = (lane & lane_mask) != 0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const float p = __shfl_xor_sync(0xffffffffu, v[i], lane_mask);
        v[i] = upper ? (p - v[i]) : (v[i] + p);
    }
}

__device__ __forceinline__ float inv_sqrt_g(int g) {
    return g == 32 ? 0.17677669529663687f : g == 64 ? 0.125f : g == 128 ? 0.08838834764831845f : g == 256 ? 0.0625f : 1.0f;
}

// ---------------------------------------------------------------- transform operand of the tensor-core RHT
// bf16 entry (n, k) of the transform operand, stored N x K (K-major): T[k][n] = S_k H_g[k][n] inside a g-chunk.
// g = 256 (Sylvester: H_256 = [[H_128, H_128], [H_128, -H_128]]): entry (n, k) of the half-transform h, T_h[k][n] =
// S_{128 h + k} H_128[k][n] / 16; the epilogue combines u = A_lo T_0 and v = A_hi T_1 into u + v and u - v.
__device__ __forceinline__ uint32_t transform_entry_256(int n, int k, const uint32_t (&sign)[4]) {
    const uint32_t neg = ((sign[k >> 5] >> (k & 31)) ^ (uint32_t)__popc(k & n)) & 1u;
    return 0x3D80u | (neg << 15);                                         // 1/16 = exact 1/sqrt(256)
}

__device__ __forceinline__ uint32_t transform_entry(int n, int k, int g, const uint32_t (&sign)[4]) {
    if ((n ^ k) & ~(g - 1)) return 0u;                                   // different g-chunks
    const int kk = k & (g - 1);
    const uint32_t neg = ((sign[kk >> 5] >> (kk & 31)) ^ (uint32_t)__popc(k & n & (g - 1))) & 1u;
    const uint32_t mag = g == 64 ? 0x3E00u : 0x3F80u;                    // 1/8 (exact 1/sqrt(64)) or 1
    return mag | (neg << 15);
}

// ---------------------------------------------------------------- scale rule and encoders
// 2^k as fp32 for k in [-149, 127] (subnormal results included).
__device__ __forceinline__ float pow2f_wide(int k) {
    return k >= -126 ? __uint_as_float((uint32_t)(k + 127) << 23) : __uint_as_float(1u << (k + 149));
}

// Algorithm 1/2 lines 1-2 for MXFP4: shared_exp = floor(log2 amax) - 2 clamped to [-127, 127];
// E8M0 byte = shared_exp + 127 = max(biased exponent of amax - 2, 0); 255 when amax is not finite.
__device__ __forceinline__ uint32_t e8m0_from_amax(float amax) {
    const uint32_t ef = __float_as_uint(amax) >> 23;          // amax >= 0
    return ef == 255u ? 255u : (ef > 2u ? ef - 2u : 0u);
}

// cvt.rn.satfinite.e2m1x2.f32: two floats -> one byte, `lo` in the low nibble; nearest-even, saturating at 6.
__device__ __forceinline__ uint32_t cvt_e2m1x2_rn(float lo, float hi) {
    uint16_t out;
    asm("{\n\t.reg .b8 b;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b, %1, %2;\n\t"
        "cvt.u16.u8 %0, b;\n\t}"
        : "=h"(out) : "f"(hi), "f"(lo));
    return out;
}

// Generic (any scale exponent) SR encoder of one value on the fp32 bit pattern.  |y| / X is formed exactly in two
// power-of-two steps, then truncated onto a grid of 2^-23 by one round-toward-zero multiply with 3/4 * 2^-126.
// That factor places E2M1's subnormal/normal boundary (1.0) on fp32's, so bits >> 22 is the E2M1 code of the lower
// neighbour and the low 22 bits are floor(frac 2^22); adding (255 - r) 2^14 + 2^13 carries into bit 22 exactly
// when 256 frac >= r + 1/2.  Truncation keeps the decision exact because the thresholds are integers there.
__device__ __forceinline__ uint32_t sr_encode_wide(float y, float p1, float p2, uint32_t r) {
    const float a = __fmul_rz(fabsf(y) * p1 * p2, __uint_as_float(0x00600000u));      // 3/4 * 2^-126
    const uint32_t t = __float_as_uint(a) + (((r ^ 0xFFu) << 14) | 0x2000u);
    return (t >> 22) | ((__float_as_uint(y) >> 28) & 8u);
}

// cvt.rz.f16x2.f32: two floats -> packed halves (lo in the low 16 bits), both truncated toward zero.
__device__ __forceinline__ uint32_t cvt_f16x2_rz(float lo, float hi) {
    uint32_t d;
    asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// cvt.rs.satfinite.e2m1x4.f32: four floats -> four E2M1 codes (v0 in the low nibble), rounded stochastically between
// grid neighbours with a 16-bit dither per value taken from `rbits` (bytes b0..b3, low to high): round up iff
// floor(65536 frac) + R >= 65536, where v0 uses R = 256 b2 + b0, v1 the same 16 bits reversed, v2 R = 256 b3 + b1 and
// v3 that one reversed.  The sign is kept (a negative value may give -0), |v| >= 6 gives 6.
__device__ __forceinline__ uint32_t cvt_e2m1x4_rs(float v0, float v1, float v2, float v3, uint32_t rbits) {
    uint16_t d;
    asm("cvt.rs.satfinite.e2m1x4.f32 %0, {%1, %2, %3, %4}, %5;" : "=h"(d) : "f"(v3), "f"(v2), "f"(v1), "f"(v0), "r"(rbits));
    return d;
}

// Two products with one factor in one instruction (mul.f32x2): each rounded like the scalar one, toward zero / to nearest.
__device__ __forceinline__ void mul2_rz(float a0, float a1, float c, float& d0, float& d1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %4};\n\tmul.rz.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(c));
}
__device__ __forceinline__ void mul2_rn(float a0, float a1, float c, float& d0, float& d1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %4};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(c));
}

// (a & ~mask) | (b & mask) in one LOP3.
__device__ __forceinline__ uint32_t bitselect(uint32_t a, uint32_t b, uint32_t mask) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xD8;" : "=r"(d) : "r"(a), "r"(b), "r"(mask));
    return d;
}

// Pipe balance: on this SM the integer/logic pipe issues a warp every other cycle while the FMA pipe (which also
// executes IMAD) issues every cycle.  `k` carries two constants the compiler must not see (they arrive as kernel
// parameters), so that the lane arithmetic below stays two multiply-adds instead of shift/add chains.
struct PipeConsts {
    uint32_t eight;    // 8
    uint32_t neg16;    // 0xFFFFFFF0
};
__host__ __device__ inline PipeConsts make_pipe_consts() { return PipeConsts{8u, 0xFFFFFFF0u}; }

// Quantise 32 consecutive fp32 values (one MX block) to 16 bytes of packed E2M1 codes + one E8M0 byte.
//   SR (Algorithm 2): round up iff 256 frac >= r + 1/2 (Eq. 2 with an 8-bit dither), decided on the exact real
//     w = (3/4) y / X.  Fast path: z = RZ(y * 3/4 * 2^(-e-14)) is truncated to fp16, two values per cvt.  The
//     factor 2^-14 places E2M1's subnormal/normal boundary on fp16's, so each 16-bit lane reads
//         s 000 ccc fffffffff      ccc = E2M1 code of the lower neighbour, f = floor(512 frac).
//     The lane is multiplied by 8 (0 ccc fffffffff 000; the sign falls into dead low bits of the next lane) and
//     8 (511 - 2r) is added: the carry into ccc is set exactly when f >= 2r + 1, i.e. 256 frac >= r + 1/2.  Both
//     truncations are toward zero and every threshold is a multiple of the fp16 spacing, so the decision is that
//     of the exact real.  One 32-bit multiply-add handles two lanes; re-inserting the sign bits from the cvt
//     result leaves the finished 4-bit code s ccc in the top nibble of each lane, so eight codes are gathered
//     with two byte permutes, one shift and one select.  Lanes pair elements (i, i+2) and (i+1, i+3), which is
//     how the four draws of one Philox word split with one mask and one byte permute.
//   SR16 (ROUNDING = 2; Algorithm 2 with a 16-bit dither): z = RZ(y * 3/4 * 2^-e) goes through the stochastic-rounding
//     convert, four values and one Philox word at a time.  The truncation keeps floor(65536 frac) of the exact real
//     because every threshold (a multiple of gap / 65536) is an fp32 number at that magnitude.
//   RN (Algorithm 1): hardware nearest-even convert of y / X.
//   ROUNDING = 3: the codes of ROUNDING = 0, computed through the same convert (see there).
// `rw` holds the block's 32 SR draws (sr_draws32); it is not read when ROUNDING = 1 (RN).
// A NaN input is out of contract (the block's scale is then taken from the other values); Inf gives byte 255.
__device__ __forceinline__ void quantize_block32_rare(const float (&y)[32], uint32_t scale_byte, const uint32_t (&rw)[8],
                                                   uint32_t (&packed)[4]) {
    // scale exponent above 100 (|values| beyond 2^103) or a non-finite block
    if (scale_byte == 255u) {
        packed[0] = packed[1] = packed[2] = packed[3] = 0u;
        return;
    }
    const int e = (int)scale_byte - 127;
    const int h1 = (-e) / 2, h2 = -e - h1;                           // exact 2^-e in two steps
    const float p1 = pow2f_wide(h1), p2 = pow2f_wide(h2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t word = 0u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = 8 * q + j;
            word |= sr_encode_wide(y[i], p1, p2, (rw[i >> 2] >> (8 * (i & 3))) & 0xFFu) << (4 * j);
        }
        packed[q] = word;
    }
}

template <int ROUNDING>
__device__ __forceinline__ void quantize_block32_rw(const float (&y)[32], const uint32_t (&rw)[8],
                                                    uint32_t (&packed)[4], uint32_t& scale_byte, const PipeConsts& k) {
    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; i += 2) amax = fmaxf(amax, fmaxf(fabsf(y[i]), fabsf(y[i + 1])));
    scale_byte = e8m0_from_amax(amax);
    const int e = (int)scale_byte - 127;
    if (ROUNDING == 0) {
        if (scale_byte > 227u) {                                     // rare: keeps the common path branch-free
            quantize_block32_rare(y, scale_byte, rw, packed);
            return;
        }
        const float c = 1.5f * pow2f_wide(-e - 15);                  // 3/4 * 2^(-e-14), a normal fp32 since e <= 100
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t u[4];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {                         // four elements share one random word
                const int i = 8 * q + 4 * hh;
                const uint32_t w = rw[2 * q + hh];
                const uint32_t r_even = w & 0x00FF00FFu;                     // r_i      | r_{i+2} << 16
                const uint32_t r_odd = __byte_perm(w, 0u, 0x4341);           // r_{i+1}  | r_{i+3} << 16
                float z0, z1, z2, z3;
                mul2_rz(y[i], y[i + 1], c, z0, z1);
                mul2_rz(y[i + 2], y[i + 3], c, z2, z3);
                const uint32_t h_even = cvt_f16x2_rz(z0, z2);
                const uint32_t h_odd = cvt_f16x2_rz(z1, z3);
                const uint32_t t_even = h_even * k.eight + (r_even * k.neg16 + 0x0FF80FF8u);   // + 8 (511 - 2r) per lane
                const uint32_t t_odd = h_odd * k.eight + (r_odd * k.neg16 + 0x0FF80FF8u);
                u[hh] = bitselect(t_even, h_even, 0x80008000u);              // s ccc .... in the top nibble of each lane
                u[2 + hh] = bitselect(t_odd, h_odd, 0x80008000u);
            }
            const uint32_t ev = __byte_perm(u[0], u[1], 0x7531);             // top bytes of elements 0, 2, 4, 6
            const uint32_t od = __byte_perm(u[2], u[3], 0x7531);             // top bytes of elements 1, 3, 5, 7
            packed[q] = bitselect(ev >> 4, od, 0xF0F0F0F0u);
        }
    } else if (ROUNDING == 3) {
        // The 8-bit rule of ROUNDING = 0 through the stochastic-rounding convert (same codes): its 16-bit dither R
        // rounds up iff floor(65536 frac) + R >= 65536, and R = 256 (255 - r) + 128 turns that into
        // 65536 frac >= 256 r + 128, i.e. 256 frac >= r + 1/2.  Only the dithers of the even code positions of a
        // convert can be chosen freely (the odd ones get the bit reversal of their neighbour's), so a convert rounds
        // two values.  Two converts per four values cost more issue slots than the integer path above, but far fewer
        // registers: the g = 256 kernel, which holds two accumulators' worth of values, is faster with it.
        if (scale_byte == 255u) {
            packed[0] = packed[1] = packed[2] = packed[3] = 0u;
            return;
        }
        const float c = 1.5f * pow2f_wide(-e - 1);                   // 3/4 * 2^-e; exact also where 2^(-e-1) is subnormal
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = 8 * q;
            const uint32_t n0 = ~rw[2 * q], n1 = ~rw[2 * q + 1];     // bytes 255 - r of elements i..i+3 and i+4..i+7
            float z[8];
#pragma unroll
            for (int j = 0; j < 8; j += 2) mul2_rz(y[i + j], y[i + j + 1], c, z[j], z[j + 1]);
            // random word of a convert: bytes (b3, b2, b1, b0) = (255 - r of position 2, 255 - r of position 0, 0x80, 0x80)
            const uint32_t ca = cvt_e2m1x4_rs(z[0], z[0], z[2], z[2], __byte_perm(n0, 0x80808080u, 0x2044));   // elements i, i+2
            const uint32_t cb = cvt_e2m1x4_rs(z[1], z[1], z[3], z[3], __byte_perm(n0, 0x80808080u, 0x3144));   // elements i+1, i+3
            const uint32_t cc = cvt_e2m1x4_rs(z[4], z[4], z[6], z[6], __byte_perm(n1, 0x80808080u, 0x2044));
            const uint32_t cd = cvt_e2m1x4_rs(z[5], z[5], z[7], z[7], __byte_perm(n1, 0x80808080u, 0x3144));
            const uint32_t ev = __byte_perm(ca, cc, 0x5410);          // codes of the even elements in the low nibble of each byte
            const uint32_t od = __byte_perm(cb, cd, 0x5410);
            packed[q] = bitselect(ev, od << 4, 0xF0F0F0F0u);
        }
    } else if (ROUNDING == 2) {
        if (scale_byte == 255u) {
            packed[0] = packed[1] = packed[2] = packed[3] = 0u;
            return;
        }
        const float c = 1.5f * pow2f_wide(-e - 1);                   // 3/4 * 2^-e; exact also where 2^(-e-1) is subnormal
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = 8 * q;
            float z[8];
#pragma unroll
            for (int j = 0; j < 8; j += 2) mul2_rz(y[i + j], y[i + j + 1], c, z[j], z[j + 1]);
            const uint32_t lo = cvt_e2m1x4_rs(z[0], z[1], z[2], z[3], rw[2 * q]);
            const uint32_t hi = cvt_e2m1x4_rs(z[4], z[5], z[6], z[7], rw[2 * q + 1]);
            packed[q] = __byte_perm(lo, hi, 0x5410);
        }
    } else {
        if (scale_byte == 255u) {
            packed[0] = packed[1] = packed[2] = packed[3] = 0u;
            return;
        }
        const float inv_x = pow2f_wide(-e);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t word = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = 8 * q + 2 * j;
                float z0, z1;
                mul2_rn(y[i], y[i + 1], inv_x, z0, z1);
                word |= cvt_e2m1x2_rn(z0, z1) << (8 * j);
            }
            packed[q] = word;
        }
    }
}

// Quantise 32 consecutive fp32 values to MXINT4: integers -7..7 as E4M3 bytes (the tensor core reads them as E4M3) + one
// E8M0 byte.  Scale: the rule of Algorithms 1 / 2 with emax_elem = 2 (largest power of two among the elements is 4).
//   SR (Algorithm 2): w = (3/4) |v| / X < 6, rounded on the integer grid with the dither of Eq. 1-2 discretised to the
//     element's 8-bit draw r: up iff 256 frac >= r + 1/2.  Exactly: a = 128 |v| / X is a power-of-two scaling, one fused
//     multiply-add toward zero forms 2^23 + floor(3 a) = 2^23 + floor(512 w), and adding 511 - 2 r carries into bit 9
//     exactly when the low nine bits are at least 2 r + 1: the rounded integer stands in bits 9..11.
//   RN (Algorithm 1): nearest integer, ties to even, saturating at 7; 2^23 + a rounded to nearest holds it in its low bits.
// Four integers at a time are the selectors of one byte permute of the table of E4M3 bytes 0, 1, .. 7.
template <bool SR>
__device__ __forceinline__ void quantize_block32_int4(const float (&v)[32], const uint32_t (&rw)[8], uint32_t (&out)[8], uint32_t& scale_byte) {
    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 32; i += 2) amax = fmaxf(amax, fmaxf(fabsf(v[i]), fabsf(v[i + 1])));
    scale_byte = e8m0_from_amax(amax);
    if (scale_byte == 255u) {
#pragma unroll
        for (int i = 0; i < 8; ++i) out[i] = 0u;
        return;
    }
    const int sh = (SR ? 7 : 0) - ((int)scale_byte - 127);              // |v| 2^sh, in two exact steps
    const float p1 = pow2f_wide(sh / 2), p2 = pow2f_wide(sh - sh / 2);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint32_t sel = 0u, sign[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float y = v[4 * w + j], a = fabsf(y) * p1 * p2;
            uint32_t q;
            if (SR) q = ((__float_as_uint(__fmaf_rz(a, 3.0f, 8388608.0f)) + 511u - 2u * ((rw[w] >> (8 * j)) & 0xFFu)) >> 9) & 7u;
            else q = __float_as_uint(__fadd_rn(fminf(a, 7.0f), 8388608.0f)) & 7u;
            sel |= q << (4 * j);
            sign[j] = __float_as_uint(y);
        }
        const uint32_t s01 = __byte_perm(sign[0], sign[1], 0x0073), s23 = __byte_perm(sign[2], sign[3], 0x0073);   // top bytes
        out[w] = __byte_perm(0x44403800u, 0x4E4C4A48u, sel) | (__byte_perm(s01, s23, 0x5410) & 0x80808080u);
    }
}

// Same, drawing the block's SR bits itself; i0 = linear index of the block's first element in the K-major operand.
__device__ __forceinline__ void quantize_block32(const float (&y)[32], int rounding, uint64_t seed, uint32_t stream_tag,
                                                 uint64_t i0, uint32_t (&packed)[4], uint32_t& scale_byte) {
    uint32_t rw[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (rounding == 0) {
        sr_draws32(seed, stream_tag, i0, rw);
        quantize_block32_rw<0>(y, rw, packed, scale_byte, make_pipe_consts());
    } else if (rounding == 2) {
        sr_draws32(seed, stream_tag, i0, rw);
        quantize_block32_rw<2>(y, rw, packed, scale_byte, make_pipe_consts());
    } else {
        quantize_block32_rw<1>(y, rw, packed, scale_byte, make_pipe_consts());
    }
}

// Byte offset of the scale of (row r, 32-block k) in the tcgen05 scale-factor tiling: 128-row x 4-block
// tiles of 512 bytes, tile (r/128, k/4) at ((r/128) * n_ktiles + k/4) * 512, inside a tile
// (r % 32) * 16 + ((r % 128) / 32) * 4 + k % 4.
__host__ __device__ __forceinline__ int64_t sf_native_offset(int64_t r, int64_t k, int64_t n_ktiles) {
    return ((r >> 7) * n_ktiles + (k >> 2)) * 512 + (r & 31) * 16 + ((r & 127) >> 5) * 4 + (k & 3);
}
// The same for the first of a row's four scales in tile `tile`, row 32 quadrant + lane of it.  Tile indices fit 32 bits, byte
// offsets do not: rows are padded to 128, so an operand of few rows passes 2^23 tiles within the element limit.
__host__ __device__ __forceinline__ uint64_t sf_row_offset(uint32_t tile, uint32_t quadrant, uint32_t lane) {
    return (uint64_t)tile * 512u + lane * 16u + quadrant * 4u;
}

}  // namespace mx
