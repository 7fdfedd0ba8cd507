// lfrec.cuh -- the fixed-point form of the rescaled Wigner recurrence and its digits
// (k_lcontract_fx.cu, k_adjoint_fx.cu).
#pragma once

#include "fxdigits.cuh"

namespace sl {

// One fixed-point step Y_{l+1} = t Y_l - Y_{l-1}, t = a' x - b', |t| < 4, |Y| < 2^60.  Words
// are split where the products need no shift: a' = Ah 2^-27 + Al 2^-58, x = xh 2^-31 + xl 2^-62,
// t = th 2^-29 + tl 2^-58 and Y = Yh 2^29 + Yl with 29-bit tl, Yl >= 0.  The two low x high
// products share a 64-bit sum whose carry into the units is rounded; tl Yl (a quarter unit on
// average, like the half) is in the rounding constant.
struct LfRec {
    long long Y, Yo;
    int xh, xl;
    __device__ __forceinline__ void step(const int4 c) {
        const long long B = (long long)(((unsigned long long)(unsigned)c.w << 32) | (unsigned)c.z);
        const long long mt = (long long)c.x * xl + ((long long)c.y * xh + (1ll << 30));
        const long long t = (long long)c.x * xh + ((mt >> 31) + B);
        const int th = (int)(t >> 29), tl = (int)t & 0x1fffffff;
        const int Yh = (int)(Y >> 29), Yl = (int)Y & 0x1fffffff;
        const long long m = (long long)th * Yl + ((long long)tl * Yh + 3 * (1ll << 27));
        const long long Yn = (long long)th * Yh + ((m >> 29) - Yo);
        Yo = Y;
        Y = Yn;
    }
};

// The coefficients of one l as LfRec takes them; zero where a' + |b'| >= 4 (big), where the
// FP64 form runs.
__device__ __forceinline__ int4 lf_coef(double a, double b, bool &big) {
    big = a + fabs(b) >= 4.0;
    const long long A = big ? 0 : fx_from_double(a, 1026), B = big ? 0 : fx_from_double(-b, 1026);  // 2^58
    const int Ah = (int)((A + (1ll << 30)) >> 31);
    return make_int4(Ah, (int)(A - (long long)Ah * (1ll << 31)), (int)B, (int)(B >> 32));
}
// x in [-1, 1] as xh 2^-31 + xl 2^-62, |xl| <= 2^30
__device__ __forceinline__ void lf_set_x(LfRec &r, double x) {
    const long long X = max(min(fx_from_double(x, 1023), (1ll << 61) - 1), 1 - (1ll << 61)) * 2;
    r.xh = (int)((X + (1ll << 30)) >> 31);
    r.xl = (int)(X - (long long)r.xh * (1ll << 31));
}
// y 2^(60 - U), rounded
__device__ __forceinline__ long long lf_from_double(double y, int U) { return (fx_from_double(y, U + 1022) + 2) >> 2; }
// |y| < 2^U for every ring and l of (m, k): |d| < 1 (but for l = 0), c falls with l, and
// cmin = min(c_L, c_{L-1}) >= 2^(ex - 1023)
__device__ __forceinline__ int lf_bound(double cmin) { return max(1, 1023 - ((__double2hiint(cmin) >> 20) & 0x7ff)); }

// Seven digits of two values Y 2^-60 in (-1, 1): fields of Y + bias at bits 52, 43, .., 7 and the
// last seven bits; a field that lies within a 16-bit half is cut from both values' halves at once.
__device__ __forceinline__ uint32_t lf_digit(uint32_t u, uint32_t mask) {
    u = (u & mask) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&u), __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500)));
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ void lf_digits(long long v0, long long v1, uint32_t d[7]) {
    constexpr unsigned long long kBias = (1ull << 60) + (1ull << 51) + (1ull << 42) + (1ull << 33) + (1ull << 24) +
                                         (1ull << 15) + (1ull << 6);
    const unsigned long long a = (unsigned long long)v0 + kBias, b = (unsigned long long)v1 + kBias;
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    const uint32_t w3 = __byte_perm(ah, bh, 0x7632), w2 = __byte_perm(ah, bh, 0x5410);
    const uint32_t w1 = __byte_perm(al, bl, 0x7632), w0 = __byte_perm(al, bl, 0x5410);
    d[0] = lf_digit(w3 >> 4, 0x03ff03ffu);
    d[1] = lf_digit(__byte_perm(ah >> 11, bh >> 11, 0x5410), 0x01ff01ffu);
    d[2] = lf_digit(w2 >> 2, 0x01ff01ffu);
    d[3] = lf_digit(__byte_perm(__funnelshift_r(al, ah, 25), __funnelshift_r(bl, bh, 25), 0x5410), 0x01ff01ffu);
    d[4] = lf_digit(w1, 0x01ff01ffu);
    d[5] = lf_digit(w0 >> 7, 0x01ff01ffu);
    d[6] = lf_digit(w0 << 2, 0x01fc01fcu);
}

}  // namespace sl
