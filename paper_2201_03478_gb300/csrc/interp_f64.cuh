// interp_f64.cuh -- the direct FP64 evaluation of one sample (step 2, Sect. 2.1):
// combined weights w_a w_b per node, the cube read through L1.
#pragma once

#include "sl_internal.cuh"

namespace sl {

template <int P>
__device__ __forceinline__ double interp_one_f64(const InterpGeom &g, const double2 *__restrict__ maps,
                                                 const StencilRec64 &r, double psi) {
    const int i = (int)(r.cell >> 16) - 1, j = (int)(r.cell & 0xffffu);
    double wt[P], wp[P];
    weights64<P>(g, i, r.dth, r.fph, wt, wp);
    int roff[P], coff[P], coffg[P];
    const unsigned ghost = stencil_offsets<P>(g, i, j, roff, coff, coffg);
    // node offsets and combined weights (ghost rows read the ring at phi + pi)
    int off[P * P];
    double w[P * P];
#pragma unroll
    for (int a = 0; a < P; ++a)
#pragma unroll
        for (int b = 0; b < P; ++b) {
            off[a * P + b] = roff[a] + (((ghost >> a) & 1u) ? coffg[b] : coff[b]);
            w[a * P + b] = wt[a] * wp[b];
            if (!SL_GUARD(off[a * P + b] >= 0 &&
                              (int64_t)off[a * P + b] + g.K < (int64_t)g.R * g.nphi * (g.K + 1),
                          0x201u))
                off[a * P + b] = 0;
        }
    double sp, cp;
    sincos(psi, &sp, &cp);
    // k = 0: only Re S_0 enters the TOD
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < P * P; ++q) acc = fma(w[q], __ldg(maps + off[q]).x, acc);
    // C_k = 2 cos(k psi), S_k = 2 sin(k psi) by the Chebyshev three-term
    // recurrence X_{k+1} = (2 cos psi) X_k - X_{k-1}
    const double c1 = 2.0 * cp;
    double Ck = c1, Sk = 2.0 * sp, Ckm = 2.0, Skm = 0.0;
    for (int k = 1; k <= g.K; ++k) {
        if (ghost) {   // (-1)^k on ghost rows: flip their weights between k-1 and k
#pragma unroll
            for (int a = 0; a < P; ++a)
                if (ghost & (1u << a))
#pragma unroll
                    for (int b = 0; b < P; ++b) w[a * P + b] = -w[a * P + b];
        }
        double sr = 0.0, si = 0.0;
#pragma unroll
        for (int q = 0; q < P * P; ++q) {
            const double2 v = __ldg(maps + off[q] + k);
            sr = fma(w[q], v.x, sr);
            si = fma(w[q], v.y, si);
        }
        acc = fma(Ck, sr, acc);
        acc = fma(-Sk, si, acc);
        const double cn = fma(c1, Ck, -Ckm), sn = fma(c1, Sk, -Skm);
        Ckm = Ck;
        Skm = Sk;
        Ck = cn;
        Sk = sn;
    }
    return acc;
}

}  // namespace sl
