// fxdigits.cuh -- 64-bit fixed point on the integer pipes and its split into
// FP16 digits for exact products on the tensor cores.
//
// GB300 runs FP64 at 1/64 of the FP32 rate (2 multiply-adds per clock and SM)
// but 1024 FP16 multiply-adds per clock and SM on mma.sync and 64 integer
// operations, so a sum of products of FP64 values is cheaper as integer digits:
//
//   x in [-1, 1] is held as X = x 2^62 (int64), rounded to 53 fraction bits and
//   split into six balanced base-512 digits,
//     x = sum_j d_j 2^(-8 - 9 j),   d_j in [-256, 256),  j = 0..5  (d_0 up to 256);
//   FP16 holds every digit exactly.  With the halves xh (digits 0..2) and xl (digits
//   3..5), x = xh 2^-26 + xl 2^-53, a sum of products is defined as
//     sum_t x_t y_t := sum_t [xh yh 2^-52 + (xh yl + xl yh) 2^-79]
//   (xl yl, below 2^-54, is left out) and computed exactly, in one of two ways with the
//   same bits:
//     - on the tensor cores, digit by digit: sum_s 2^(-16 - 9 s) acc_s, s = 0..7,
//       acc_s = sum_t sum_{i + j = s} dx_i dy_j over the 27 pairs with i < 3 or j < 3.
//       With at most 32 terms t, |acc_s| <= 6 x 32 x 2^16 < 2^24: the FP32
//       accumulators of the MMA hold it exactly, whatever the order of the terms;
//     - on the integer pipe, three 32 x 32 + 64 bit multiply-adds per term (fx_split).
//   The operands' rounding (2^-54 each) and xl yl remain, the size of one FP64 rounding
//   of the largest product.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "fxint.cuh"

namespace sl {

constexpr int kFxDig = 6, kFxSums = 8;
// half a unit of the last digit (2^8) plus 256 in every digit: makes the digits
// of X + bias unsigned 9-bit fields (10 bits for the first)
constexpr unsigned long long kFxBias = (1ull << 62) + (1ull << 53) + (1ull << 44) + (1ull << 35) + (1ull << 26) +
                                       (1ull << 17) + (1ull << 8);
// Digits for operands of twice the range: x in (-2 + 2^-8, 2 - 2^-8), X = x 2^62, d_0 within
// +-512, which FP16 and the sums above still hold (32 x (5 x 2^16 + 2^17) < 2^24).
constexpr unsigned long long kFxBiasWide = kFxBias + (1ull << 62);

// digit pairs (a's digit in the low half, b's in the high half) of two Q62 values:
// the 9-bit field u goes into the mantissa of FP16 1024 + u, minus 1280
__device__ __forceinline__ uint32_t fx_field(uint32_t a, uint32_t b, uint32_t mask, unsigned short offset = 0x6500) {
    const uint32_t u = (__byte_perm(a, b, 0x5410) & mask) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&u), __halves2half2(__ushort_as_half(offset), __ushort_as_half(offset)));
    return *reinterpret_cast<const uint32_t *>(&h);
}
// N = 6: rounded to 53 fraction bits; N = 7: a seventh digit 2^-62 takes what the six leave over (exact)
template <bool WIDE = false, int N>
__device__ __forceinline__ void fx_digits(long long a, long long b, uint32_t (&d)[N]) {
    static_assert(N == kFxDig || N == kFxDig + 1, "six digits or seven");
    constexpr unsigned long long kBias = WIDE ? kFxBiasWide : kFxBias;
    const unsigned long long ya = (unsigned long long)a + kBias, yb = (unsigned long long)b + kBias;
    const uint32_t ah = (uint32_t)(ya >> 32), al = (uint32_t)ya, bh = (uint32_t)(yb >> 32), bl = (uint32_t)yb;
    d[0] = fx_field(ah >> 22, bh >> 22, 0x03ff03ffu, WIDE ? 0x6600 : 0x6500);   // minus 1536 or 1280
    d[1] = fx_field(ah >> 13, bh >> 13, 0x01ff01ffu);
    d[2] = fx_field(ah >> 4, bh >> 4, 0x01ff01ffu);
    d[3] = fx_field(__funnelshift_r(al, ah, 27), __funnelshift_r(bl, bh, 27), 0x01ff01ffu);
    d[4] = fx_field(al >> 18, bl >> 18, 0x01ff01ffu);
    d[5] = fx_field(al >> 9, bl >> 9, 0x01ff01ffu);
    if constexpr (N > kFxDig) d[6] = fx_field(al, bl, 0x01ff01ffu);
}

// x 2^(Q - e) (truncated toward zero below the unit) for |x| < 2^e, e = ef - 1022, by
// its bits; ef: the largest biased exponent among the values sharing the scale,
// 64 <= ef < 2047.  Values 2^64 times smaller than the scale give 0.
template <int Q = 62>
__device__ __forceinline__ long long fx_from_double(double x, int ef) {
    static_assert(Q == 62 || Q == 63, "sign bit left");
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    const int sh = min(ef - ex, 63);
    const unsigned long long m = (((b & ((1ull << 52) - 1)) | (1ull << 52)) << (Q - 53)) >> sh;
    const long long sg = (long long)b >> 63;
    return ((long long)m ^ sg) - sg;
}

// c += A B on 16 x 8 x 16 FP16 fragments (c = A B with first)
__device__ __forceinline__ void mma_f16(float &c0, float &c1, float &c2, float &c3, const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1, bool first = false) {
    if (first)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
            : "=f"(c0), "=f"(c1), "=f"(c2), "=f"(c3)
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(c0), "+f"(c1), "+f"(c2), "+f"(c3)
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c += A B on 16 x 8 x 8 FP16 fragments
__device__ __forceinline__ void mma_f16_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(b));
}

// xh (digits 0..2) and xl (digits 3..5) of a Q62 value
template <bool WIDE = false>
__device__ __forceinline__ void fx_split(long long x, int &h, int &l) {
    constexpr int kBias27 = (1 << 26) + (1 << 17) + (1 << 8);       // 256 in each of three digits
    const unsigned long long y = (unsigned long long)x + (WIDE ? kFxBiasWide : kFxBias);
    h = (int)(uint32_t)(y >> 36) - kBias27 - (WIDE ? 1 << 26 : 0);
    l = (int)((uint32_t)(y >> 9) & 0x7ffffffu) - kBias27;
}

// The product sum times 2^57, rounded: from the digit sums (orders 0 to 7, or 0 to 6 and
// rounded to even: with one factor 1 a 32nd of the sums are ties), and from sum xh yh and
// sum (xh yl + xl yh).
template <int N>
__device__ __forceinline__ long long fx_combine(const float (&a)[N]) {
    static_assert(N == kFxSums || N == kFxSums - 1, "orders 0 to 7 or 0 to 6");
    long long v;
    if constexpr (N == kFxSums) {
        long long x = (long long)__float2int_rn(a[7]) + (1ll << 21);
        x += (long long)__float2int_rn(a[6]) * 512ll;
        x += (long long)__float2int_rn(a[5]) * 262144ll;
        v = x >> 22;
    } else {
        v = fx_shift_even((long long)__float2int_rn(a[6]) + (long long)__float2int_rn(a[5]) * 512ll, 13);
    }
    v += (long long)__float2int_rn(a[4]) * 32ll;
    v += (long long)__float2int_rn(a[3]) * 16384ll;
    v += (long long)__float2int_rn(a[2]) * 8388608ll;
    v += (long long)((unsigned long long)(uint32_t)(__float2int_rn(a[1]) + __float2int_rn(a[0]) * 512) << 32);
    return v;
}
__device__ __forceinline__ long long fx_combine(long long hh, long long x) { return hh * 32 + ((x + (1ll << 21)) >> 22); }

// (cos, sin)(psi) in Q62 by fixed-point arithmetic, |error| < 2^-57, for |psi| < 2^9;
// false otherwise (and for NaN).  The 53-bit mantissa times 1/(2 pi) to 128 bits gives
// psi in turns to 2^-64; the nearest of 256 table angles (tab[i] = (cos, sin)(2 pi i / 256),
// Q62) is rotated by the rest, |delta| <= pi / 256, through
//   sin delta = delta (1 - t (1/6 - t (1/120 - t / 5040))),  cos delta = 1 - t (1/2 - t (1/24 - t / 720)),
// t = delta^2 (the next terms are below 2^-62).  In FP64 this is 45 operations at 1/64
// of the FP32 rate.
__device__ __forceinline__ bool fx_sincos(double psi, const longlong2 *tab, long long &c, long long &s) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(psi);
    const int e = ((int)(bits >> 52) & 0x7ff) - 1023;
    c = kFxOne;
    s = 0;
    if (e > 8) return false;
    if (e < -62) return true;
    // 1 / (2 pi) 2^128 = (chi : clo)
    constexpr unsigned long long chi = 0x28be60db9391054aull, clo = 0x7f09d5f47d4d3770ull;
    const unsigned long long M = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const unsigned long long l = M * chi, h0 = __umul64hi(M, chi), p1 = l + __umul64hi(M, clo);
    const unsigned long long p2 = h0 + (p1 < l ? 1ull : 0ull);
    // turns = (p2 : p1) 2^(e - 116) (the low word dropped): 64 fraction bits from bit 52 - e
    const int sh = 52 - e;                                   // in [44, 114]
    unsigned long long u = sh < 64 ? ((p1 >> sh) | (p2 << (64 - sh))) : (p2 >> (sh - 64));
    if (bits >> 63) u = 0ull - u;
    const unsigned long long ur = u + (1ull << 55);
    const longlong2 cs = tab[(unsigned)(ur >> 56)];
    const long long R = (long long)((ur << 8) ^ (1ull << 63));       // rest in turns, times 2^72
    const long long d = __mul64hi(R, 0x6487ed5110b4611all);          // delta, Q68 (2 pi / 16 2^64)
    const long long t = fx_mulhi(d, d);                              // Q72
    const long long qs = 768614336404564651ll - fx_mulhi(t, 150119987579017ll - fx_mulhi(t, 13962052416ll));
    const long long qc = (1ll << 61) - fx_mulhi(t, 750599937895083ll - fx_mulhi(t, 97734366913ll));
    const long long sd = (d - (fx_mulhi(d, fx_mulhi(t, qs)) >> 6)) >> 6;     // sin delta, Q62
    const long long vd = fx_mulhi(t, qc) >> 8;                               // 1 - cos delta
    c = cs.x - fx_mul(cs.x, vd) - fx_mul(cs.y, sd);
    s = cs.y + fx_mul(cs.x, sd) - fx_mul(cs.y, vd);
    return true;
}

}  // namespace sl
