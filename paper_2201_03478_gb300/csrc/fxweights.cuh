// fxweights.cuh -- interpolation weights of the fixed-point kernels (k_interp_fx.cu,
// k_interp_adj_fx.cu).
#pragma once

#include "sl_internal.cuh"

namespace sl {

// phi weights of the fraction f in [0, 1): at p = 4 with a = f (f - 1) and b = a - 2 =
// (f + 1)(f - 2), 8 FP64 operations instead of 15
template <int P>
__device__ __forceinline__ void fx_phi_weights(double f, double wp[P]) {
    if constexpr (P == 4) {
        const double a = fma(f, f, -f), a6 = a * (1.0 / 6.0), b2 = fma(0.5, a, -1.0);
        wp[0] = fma(-a6, f, a6 + a6);
        wp[1] = fma(b2, f, -b2);
        wp[2] = -b2 * f;
        wp[3] = fma(a6, f, a6);
    } else {
        lagrange_phi<P>(f, wp);
    }
}

// theta and phi weights of one sample in FP64
template <int P>
__device__ __forceinline__ void fx_weights(const InterpGeom &g, int i, double dth, double fph, double wt[P], double wp[P]) {
    double o[P], wd[P];
#pragma unroll
    for (int a = 0; a < P; ++a) {
        o[a] = __ldg(g.offs64 + (size_t)(i + 1) * P + a);
        wd[a] = __ldg(g.wden + (size_t)(i + 1) * P + a);
    }
    lagrange_theta<P>(dth, o, wd, wt);
    fx_phi_weights<P>(fph, wp);
}

// x of [-2, 2] in Q62; false when |x| >= 2 or x is NaN
__device__ __forceinline__ bool fx_q62(double x, long long &v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    if (ex >= 1024) return false;
    const int sh = 1023 - ex;                        // value = m 2^(ex - 1075), times 2^62
    const unsigned long long m0 = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const unsigned long long m = (m0 << 10) >> min(sh, 63);
    const long long sg = (long long)b >> 63;
    v = ((long long)m ^ sg) - sg;
    return true;
}

}  // namespace sl
