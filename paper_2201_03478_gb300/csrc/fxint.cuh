// fxint.cuh -- the 64-bit integer arithmetic of the fixed-point kernels.  Plain C++ (it also compiles
// without nvcc, for tests on the host); sums that may pass 2^63 before the next term brings them back
// are formed unsigned, where wrapping is defined.
#pragma once

#ifdef __CUDACC__
#define SL_FX_FN __device__ __forceinline__
#else
#define SL_FX_FN static inline
#endif

namespace sl {

constexpr long long kFxOne = 1ll << 62;

// (a b) 2^-64 for |a|, |b| <= 2^62, at most two units off: the product of the low
// halves is left out, and halves signed by a carry into the high ones keep all
// three partial products signed 32 x 32 multiply-adds
SL_FX_FN long long fx_mulhi(long long a, long long b) {
    const int al = (int)a, bl = (int)b;
    const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31), bh = (int)(b >> 32) + (int)((unsigned)bl >> 31);
    const long long m = (long long)ah * bl + (long long)bh * al;
    return (long long)ah * bh + (m >> 32);
}
// the same rounded to nearest; |a| < 2^62.6 with |b| <= 1.5 x 2^62 is in range too
SL_FX_FN long long fx_mulhi_rn(long long a, long long b) {
    const int al = (int)a, bl = (int)b;
    const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31), bh = (int)(b >> 32) + (int)((unsigned)bl >> 31);
    const long long m = (long long)ah * bl + ((long long)bh * al + (1ll << 31));
    return (long long)ah * bh + (m >> 32);
}
// a b for Q62 operands (|a|, |b| <= 1): Q62, at most 2^-59 off
SL_FX_FN long long fx_mul(long long a, long long b) {
    return (long long)((unsigned long long)fx_mulhi(a, b) << 2);
}
// the same rounded to nearest, without the truncation's bias (zero stays zero): at most 2^-61 off
SL_FX_FN long long fx_mul_rn(long long a, long long b) {
    const int al = (int)a, bl = (int)b;
    const int ah = (int)(a >> 32) + (int)((unsigned)al >> 31), bh = (int)(b >> 32) + (int)((unsigned)bl >> 31);
    const long long m = (long long)ah * bl + (long long)bh * al;
    return (long long)ah * bh * 4 + ((m + (1ll << 29)) >> 30);
}
// 2 c x - p in Q62 (|c|, |x|, |p| <= 1): one step of X_{k+1} = 2 cos(a) X_k - X_{k-1}; at c = x = 1 the
// product alone is 2^63
SL_FX_FN long long fx_cheb(long long c, long long x, long long p) {
    return (long long)(((unsigned long long)fx_mulhi(c, x) << 3) - (unsigned long long)p);
}

// x 2^-n rounded to nearest, ties to even
SL_FX_FN long long fx_shift_even(long long x, int n) {
    return n > 0 ? (x + ((1ll << (n - 1)) - 1) + ((x >> n) & 1)) >> n : x;
}

}  // namespace sl
