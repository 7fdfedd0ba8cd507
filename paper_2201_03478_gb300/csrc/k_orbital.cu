// k_orbital.cu -- the orbital dipole and quadrupole seen through the full 4pi
// beam (Sect. 3.3, Eqs. dipole and dipole_fast), with the paper's acceleration:
// the rotation into the beam frame at every s-th sample of a pointing period,
// a cubic spline in between, and the remainder of each period exact.
//
//   D~ = T0 [ S . beta' + q beta'^T S2 beta' ],   beta' = R^T beta,
//   R = Rz(phi) Ry(theta) Rz(psi)  (the beam-to-sky rotation of Sect. 2.1),
//
// with S = (S_x, S_y, S_z) and S2 the symmetric matrix of S_xx ... S_yz: the
// moments int v B dOmega of the temperature beam in its own frame.  Only the
// l <= 2 beam coefficients enter them (closed forms in k_orb_moments).
//
// Kernels (all FP64):
//   k_orb_moments  one thread: the nine moments from b_lk, l <= 2
//   k_orb_nodes    one thread per spline node: Eq. dipole_fast at that sample
//   k_orb_spline   one CTA per pointing period (a warp for short ones, k_orb_spline_tiny's
//                  threads for the shortest): the cubics of the natural spline through
//                  the period's nodes
//   k_orb_eval     one thread per sample: the cubic between nodes, Eq.
//                  dipole_fast after the last node (or everywhere when s = 1)
// All are bound by the FP64 pipe (2 operations a clock and SM), so they keep its work
// small: sines and cosines in 64-bit fixed point on the integer pipe (fx_sincos; absolute
// error 2^-57, below the products' rounding), three multiply-adds a sample in the cubic.
// 4e7 samples, s = 20 (nodes, spline, evaluation): 391, 155, 332 -> 154, 119, 274 us.
//
// The spline system N_{j-1} + 4 N_j + N_{j+1} = y_{j+1} - 2 y_j + y_{j-1} (N = M s^2 / 6, M the
// second derivatives, M_0 = M_{n-1} = 0) is solved by the tridiagonal elimination
//   dp_j = (rhs_j - dp_{j-1}) c_j,  N_j = dp_j - c_j N_{j+1},  c_j = 1 / (4 - c_{j-1}),
// whose pivots c_j reach their limit 2 - sqrt(3) (to the last bit) within
// kOrbPivots rows.  Both sweeps are first-order recurrences d' = a - c d, affine in the value
// before, so a thread runs kOrbRun rows from zero, the threads' maps (end value from zero, factor)
// are combined by a scan, and each thread adds its rows' share of the value that enters it.
// |c| <= 0.268: the factor of 64 rows (0.268^64 < 1e-36) is below any rounding, so the scan
// combines 8 threads, and what enters a warp is the end value of the warp before.
//
// Between nodes j and j + 1 the spline is c0 + B (c1 + B (c2 + B c3)), B = r / s (a table),
// r = t - j s, with c0 = y_j, c1 = y_{j+1} - y_j - (2 N_j + N_{j+1}), c2 = 3 N_j,
// c3 = N_{j+1} - N_j.
#include <cmath>

#include "fxdigits.cuh"
#include "sl_internal.cuh"

namespace sl {

constexpr int kOrbEvalPerThread = 8;   // samples per thread of k_orb_eval
constexpr int kOrbRun = 8;             // rows per thread and sweep round of k_orb_spline
constexpr int kOrbPivots = 40;         // pivots tabulated; the last one is the limit

// x 2^-62, x = 0 or |x| >= 1: the exponent lowered by integer arithmetic
__device__ __forceinline__ double orb_q62(long long x) {
    const double v = (double)x;
    return x ? __hiloint2double(__double2hiint(v) - (62 << 20), __double2loint(v)) : 0.0;
}
__device__ __forceinline__ void orb_sincos(double x, const longlong2 *tab, double &s, double &c) {
    long long fc, fs;
    if (fx_sincos(x, tab, fc, fs)) {
        s = orb_q62(fs);
        c = orb_q62(fc);
    } else {                                     // |x| >= 2^9 or not finite
        sincos(x, &s, &c);
    }
}

// Eq. dipole_fast at one sample.  beta' = Rz(-psi) Ry(-theta) Rz(-phi) beta.
__device__ __forceinline__ double orb_value(const longlong2 *tab, const double *__restrict__ S, double T0, double q,
                                            double th, double ph, double ps, const double *__restrict__ b) {
    double st, ct, sp, cp, ss, cs;
    orb_sincos(th, tab, st, ct);
    orb_sincos(ph, tab, sp, cp);
    orb_sincos(ps, tab, ss, cs);
    const double u = cp * b[0] + sp * b[1];      // Rz(-phi)
    const double v = -sp * b[0] + cp * b[1];
    const double x1 = ct * u - st * b[2];        // Ry(-theta)
    const double z = st * u + ct * b[2];
    const double x = cs * x1 + ss * v;           // Rz(-psi)
    const double y = -ss * x1 + cs * v;
    const double lin = S[0] * x + S[1] * y + S[2] * z;
    const double quad = S[3] * x * x + S[4] * y * y + S[5] * z * z +
                        2.0 * (S[6] * x * y + S[7] * x * z + S[8] * y * z);
    return T0 * (lin + q * quad);
}

// The nine moments of the temperature beam (component 0 of [ncomp][K+1][L+1]).
// Writing each v in spherical harmonics (Condon-Shortley phase) and using
// b_{l,-m} = (-1)^m conj(b_lm):  z = sqrt(4pi/3) Y10, x + iy = -sqrt(8pi/3) Y11,
// 1 = sqrt(4pi) Y00, z^2 = sqrt(4pi)/3 Y00 + (4/3) sqrt(pi/5) Y20,
// (x + iy)^2 = sqrt(32pi/15) Y22, (x + iy) z = -sqrt(8pi/15) Y21.
__global__ void k_orb_moments(const double2 *__restrict__ beam, int L, int K, double *__restrict__ S) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto b = [&](int l, int k) -> double2 {
        return (l <= L && k <= K && k <= l) ? beam[(int64_t)k * (L + 1) + l] : make_double2(0.0, 0.0);
    };
    const double pi = 3.14159265358979323846;
    const double b00 = b(0, 0).x, b10 = b(1, 0).x, b20 = b(2, 0).x;
    const double2 b11 = b(1, 1), b21 = b(2, 1), b22 = b(2, 2);
    const double mono = sqrt(4.0 * pi) / 3.0 * b00;
    const double c22 = sqrt(32.0 * pi / 15.0), c21 = sqrt(8.0 * pi / 15.0), c20 = sqrt(pi / 5.0);
    S[0] = -2.0 * sqrt(2.0 * pi / 3.0) * b11.x;
    S[1] = 2.0 * sqrt(2.0 * pi / 3.0) * b11.y;
    S[2] = sqrt(4.0 * pi / 3.0) * b10;
    S[3] = mono - 2.0 / 3.0 * c20 * b20 + 0.5 * c22 * b22.x;
    S[4] = mono - 2.0 / 3.0 * c20 * b20 - 0.5 * c22 * b22.x;
    S[5] = mono + 4.0 / 3.0 * c20 * b20;
    S[6] = -0.5 * c22 * b22.y;
    S[7] = -c21 * b21.x;
    S[8] = c21 * b21.y;
}

struct OrbArgs {
    const double *theta, *phi, *psi;
    const int64_t *start;     // [nper + 1] first sample of each period
    const int64_t *noff;      // [nper + 1] first node of each period
    const double *beta;       // [nper][3]
    const double *S;          // [9]
    const double *piv;        // [kOrbPivots] c_j (c_0 = 0); c_j = piv[kOrbPivots - 1] beyond
    const double *frac;       // [s + 1] r / s
    const longlong2 *tab;     // (cos, sin)(2 pi i / 256), Q62
    double T0, q;
    int64_t n, nper, nnodes;
    int s;
    double *y;                // [nnodes] node values
    double4_32a *cub;         // [nnodes] cubics from each node on
    double *tod;
    int accumulate;
};

// largest p in [lo, hi) with v[p] <= x, given v[lo] <= x < v[hi]
__device__ __forceinline__ int64_t orb_find(const int64_t *__restrict__ v, int64_t lo, int64_t hi, int64_t x) {
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (v[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(256) k_orb_nodes(const OrbArgs a) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < a.nnodes;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = orb_find(a.noff, 0, a.nper, g);
        const int64_t i = a.start[p] + (int64_t)a.s * (g - a.noff[p]);
        a.y[g] = orb_value(a.tab, a.S, a.T0, a.q, a.theta[i], a.phi[i], a.psi[i], a.beta + 3 * p);
    }
}

// shared-memory slot of round row q: one pad slot per thread's run, so that the lanes'
// rows (8 l + i) fall on distinct banks
__device__ __forceinline__ int orb_pad(int q) { return q + (q >> 3); }
// threads per period: one warp up to kOrbShortNodes nodes (one round of it), eight beyond.  A short
// period leaves most of eight warps at barriers: 1e7 samples in periods of 1950 (98 nodes, s = 20) 97 -> 51
// us, of 4000 (200 nodes) 58 -> 30.  The shortest: k_orb_spline_tiny.
constexpr int kOrbThreads = 256, kOrbShortThreads = 32;

// The value that enters this thread's rows, from every thread's (end value from zero A, factor F)
// and the value that enters the round; ends[warp]: the warps' end values (the last one the round's).
__device__ __forceinline__ double orb_enter(double A, double F, double carry, double *ends) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const double pa = __shfl_up_sync(0xffffffffu, A, o), pf = __shfl_up_sync(0xffffffffu, F, o);
        if (lane >= o) {
            A = fma(F, pa, A);
            F *= pf;
        }
    }
    if (lane == 31) ends[warp] = A;
    __syncthreads();
    const double in = warp ? ends[warp - 1] : carry;
    const double pa = __shfl_up_sync(0xffffffffu, A, 1), pf = __shfl_up_sync(0xffffffffu, F, 1);
    return lane ? fma(pf, in, pa) : in;
}

// One CTA of NT threads per period: both sweeps in rounds of NT x kOrbRun rows, values staged through shared
// memory so that global accesses are coalesced.  The forward sweep's dp_j wait in the first
// quarter of the period's cubics: cubic j (doubles 4 j .. 4 j + 3) replaces dp values of rows at
// or above j, which the backward sweep has read by then.
template <int NT>
__global__ void __launch_bounds__(NT) k_orb_spline(const OrbArgs a) {
    constexpr int ROUND = NT * kOrbRun, PAD = ROUND + ROUND / kOrbRun + 2;
    __shared__ double s_piv[kOrbPivots];
    __shared__ double s_y[PAD], s_d[PAD];
    __shared__ double s_end[2][NT / 32];
    const int64_t p = blockIdx.x;
    const int64_t g0 = a.noff[p], M = a.noff[p + 1] - g0;
    if (M <= kOrbTinyNodes || (M <= kOrbShortNodes) != (NT == kOrbShortThreads)) return;    // nothing to do, or another launch's
    for (int j = threadIdx.x; j < kOrbPivots; j += NT) s_piv[j] = a.piv[j];
    __syncthreads();
    const double *__restrict__ y = a.y + g0;
    double4_32a *cub = a.cub + g0;
    double *dp = reinterpret_cast<double *>(cub);
    auto piv = [&](int64_t j) { return s_piv[j < kOrbPivots ? j : kOrbPivots - 1]; };
    const int lo = threadIdx.x * kOrbRun;
    int par = 0;                                     // s_end is used alternately: one barrier a round less
    // forward sweep over rows 1 .. M-2: dp_j = (rhs_j - dp_{j-1}) c_j, dp_0 = 0
    double carry = 0.0;
    for (int64_t base = 1; base <= M - 2; base += ROUND, par ^= 1) {
        const int rows = (int)min((int64_t)ROUND, M - 1 - base);
        for (int k = threadIdx.x; k < rows + 2; k += NT) s_y[orb_pad(k)] = y[base - 1 + k];
        __syncthreads();
        double v[kOrbRun], d = 0.0, f = 1.0;
#pragma unroll
        for (int i = 0; i < kOrbRun; ++i)
            if (lo + i < rows) {
                const int k = lo + i;
                const double c = piv(base + k);
                d = (s_y[orb_pad(k + 2)] - 2.0 * s_y[orb_pad(k + 1)] + s_y[orb_pad(k)] - d) * c;
                f *= -c;
                v[i] = d;
            }
        double in = orb_enter(d, f, carry, s_end[par]);
        carry = s_end[par][NT / 32 - 1];
#pragma unroll
        for (int i = 0; i < kOrbRun; ++i)
            if (lo + i < rows) {
                in *= -piv(base + lo + i);
                s_d[orb_pad(lo + i)] = v[i] + in;
            }
        __syncthreads();
        for (int k = threadIdx.x; k < rows; k += NT) dp[base + k] = s_d[orb_pad(k)];
    }
    __syncthreads();                                 // dp is read by other threads than wrote it
    // backward sweep: N_j = dp_j - c_j N_{j+1}, N_{M-1} = 0; round row q is j = top - q, then the
    // cubics of nodes top .. top - rows + 1, from N_j and N_{j+1}
    carry = 0.0;
    double above = 0.0;                              // N of the row above the round
    for (int64_t top = M - 2; top >= 1; top -= ROUND, par ^= 1) {
        const int rows = (int)min((int64_t)ROUND, top);
        for (int k = threadIdx.x; k < rows; k += NT) s_d[orb_pad(k)] = dp[top - k];
        for (int k = threadIdx.x; k < rows + 1; k += NT) s_y[orb_pad(k)] = y[top + 1 - k];
        __syncthreads();
        double v[kOrbRun], m = 0.0, f = 1.0;
#pragma unroll
        for (int i = 0; i < kOrbRun; ++i)
            if (lo + i < rows) {
                const double c = piv(top - lo - i);
                m = s_d[orb_pad(lo + i)] - c * m;
                f *= -c;
                v[i] = m;
            }
        double in = orb_enter(m, f, carry, s_end[par]);
        carry = s_end[par][NT / 32 - 1];
#pragma unroll
        for (int i = 0; i < kOrbRun; ++i)
            if (lo + i < rows) {
                in *= -piv(top - lo - i);
                s_d[orb_pad(lo + i)] = v[i] + in;
            }
        __syncthreads();
        for (int k = threadIdx.x; k < rows; k += NT) {
            const double m0 = s_d[orb_pad(k)], m1 = k ? s_d[orb_pad(k - 1)] : above;
            const double y0 = s_y[orb_pad(k + 1)], y1 = s_y[orb_pad(k)];
            cub[top - k] = make_double4_32a(y0, (y1 - y0) - fma(2.0, m0, m1), 3.0 * m0, m1 - m0);
        }
        above = s_d[orb_pad(rows - 1)];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double m1 = above;                     // node 0: N_0 = 0, N_1 (0 when there are two nodes)
        cub[0] = make_double4_32a(y[0], (y[1] - y[0]) - m1, 0.0, m1);
    }
}

// The same for periods of 2 to kOrbTinyNodes nodes, a thread each, row by row: in a warp of its own such a
// period leaves most lanes of every FP64 instruction empty: 5e6 samples in periods of 50, s = 7 (8 nodes) 564 ->
// 22 us, of 200, s = 12 (17 nodes) 180 -> 18; at 25 nodes 1e6 samples take the warp form's 77 us.
constexpr int kOrbTinyThreads = 128;

__global__ void __launch_bounds__(kOrbTinyThreads) k_orb_spline_tiny(const OrbArgs a) {
    static_assert(kOrbTinyNodes <= kOrbPivots, "pivots tabulated");
    __shared__ double s_piv[kOrbPivots], s_dp[kOrbTinyNodes][kOrbTinyThreads];
    for (int j = threadIdx.x; j < kOrbPivots; j += kOrbTinyThreads) s_piv[j] = a.piv[j];
    __syncthreads();
    const int64_t p = (int64_t)blockIdx.x * kOrbTinyThreads + threadIdx.x;
    if (p >= a.nper) return;
    const int64_t g0 = a.noff[p];
    if (a.noff[p + 1] - g0 < 2 || a.noff[p + 1] - g0 > kOrbTinyNodes) return;
    const int M = (int)(a.noff[p + 1] - g0);
    const double *__restrict__ y = a.y + g0;
    double4_32a *cub = a.cub + g0;
    double d = 0.0, y0 = y[0], y1 = y[1];
    for (int j = 1; j <= M - 2; ++j) {
        const double y2 = y[j + 1];
        d = (y2 - 2.0 * y1 + y0 - d) * s_piv[j];
        s_dp[j][threadIdx.x] = d;
        y0 = y1;
        y1 = y2;
    }
    double m1 = 0.0;                                 // N of the row above; y0, y1: nodes M - 2 and M - 1
    for (int j = M - 2; j >= 1; --j) {
        const double m0 = s_dp[j][threadIdx.x] - s_piv[j] * m1;
        cub[j] = make_double4_32a(y0, (y1 - y0) - fma(2.0, m0, m1), 3.0 * m0, m1 - m0);
        m1 = m0;
        y1 = y0;
        y0 = y[j - 1];
    }
    cub[0] = make_double4_32a(y0, (y1 - y0) - m1, 0.0, m1);
}

__global__ void __launch_bounds__(256) k_orb_eval(const OrbArgs a) {
    __shared__ int64_t s_p[2];
    const int64_t c0 = (int64_t)blockIdx.x * blockDim.x * kOrbEvalPerThread;
    const int64_t c1 = min(a.n, c0 + (int64_t)blockDim.x * kOrbEvalPerThread);
    if (threadIdx.x == 0) {
        s_p[0] = orb_find(a.start, 0, a.nper, c0);
        s_p[1] = orb_find(a.start, 0, a.nper, c1 - 1);
    }
    __syncthreads();
    const int64_t p0 = s_p[0], p1 = s_p[1];
    const unsigned su = (unsigned)a.s;
#pragma unroll 2
    for (int r = 0; r < kOrbEvalPerThread; ++r) {
        const int64_t i = c0 + threadIdx.x + (int64_t)r * blockDim.x;
        if (i >= c1) break;
        const int64_t p = p0 == p1 ? p0 : orb_find(a.start, p0, p1 + 1, i);
        const unsigned t = (unsigned)(i - a.start[p]);      // periods hold < 2^31 samples
        double val;
        bool exact = su == 1;
        if (!exact) {
            const int64_t g0 = a.noff[p];
            const unsigned M = (unsigned)(a.noff[p + 1] - g0);
            const unsigned jt = t / su;
            if (jt >= M || (jt == M - 1 && t != jt * su)) {
                exact = true;                                   // after the last node
            } else if (M == 1) {
                val = a.y[g0];
            } else {
                const unsigned j = jt < M - 1 ? jt : M - 2;
                if (SL_GUARD(g0 + j + 1 < a.nnodes && t - j * su <= su, 0x501u)) {
                    const double B = __ldg(a.frac + (t - j * su));      // r = t - j s (s at the last node)
                    const double4_32a c = a.cub[g0 + j];
                    val = fma(B, fma(B, fma(B, c.w, c.z), c.y), c.x);
                } else {
                    val = 0.0;
                }
            }
        }
        if (exact) val = orb_value(a.tab, a.S, a.T0, a.q, a.theta[i], a.phi[i], a.psi[i], a.beta + 3 * p);
        a.tod[i] = a.accumulate ? a.tod[i] + val : val;
    }
}

sl_status launch_orb_moments(sl_plan *p, const double *beam, double *S) {
    k_orb_moments<<<1, 32, 0, p->stream>>>((const double2 *)beam, p->L, p->K, S);
    return cuda_check(cudaGetLastError(), "k_orb_moments launch");
}

sl_status launch_orbital(sl_plan *p, const OrbLaunch &o) {
    OrbArgs a;
    a.theta = o.theta;
    a.phi = o.phi;
    a.psi = o.psi;
    a.start = o.start;
    a.noff = o.noff;
    a.beta = o.beta;
    a.S = o.S;
    a.piv = o.piv;
    a.frac = o.frac;
    a.tab = p->geom.phase_tab;
    a.T0 = o.T0;
    a.q = o.q;
    a.n = o.n;
    a.nper = o.nper;
    a.nnodes = o.nnodes;
    a.s = o.s;
    a.y = o.y;
    a.cub = reinterpret_cast<double4_32a *>(o.cub);
    a.tod = o.tod;
    a.accumulate = o.accumulate;
    int slot;
    if (a.s > 1 && a.nnodes > 0) {
        const int64_t nb = std::min<int64_t>((a.nnodes + 255) / 256, 152 * 32);
        slot = timing_begin(p, "orb_nodes");
        k_orb_nodes<<<(unsigned)nb, 256, 0, p->stream>>>(a);
        timing_end(p, slot);
        sl_status st = cuda_check(cudaGetLastError(), "k_orb_nodes launch");
        if (st != SL_OK) return st;
        slot = timing_begin(p, "orb_spline");
        if (o.ntiny > 0)
            k_orb_spline_tiny<<<(unsigned)((a.nper + kOrbTinyThreads - 1) / kOrbTinyThreads), kOrbTinyThreads, 0, p->stream>>>(a);
        if (o.nshort > 0) k_orb_spline<kOrbShortThreads><<<(unsigned)a.nper, kOrbShortThreads, 0, p->stream>>>(a);
        if (o.nlong > 0) k_orb_spline<kOrbThreads><<<(unsigned)a.nper, kOrbThreads, 0, p->stream>>>(a);
        timing_end(p, slot);
        if ((st = cuda_check(cudaGetLastError(), "k_orb_spline launch")) != SL_OK) return st;
    }
    const int64_t per_cta = 256 * kOrbEvalPerThread;
    const int64_t nb = (a.n + per_cta - 1) / per_cta;
    if (nb > 0x7fffffff) return set_error(SL_ERR_UNSUPPORTED, "orbital_dipole_tod: n too large");
    slot = timing_begin(p, a.s == 1 ? "orb_exact" : "orb_eval");
    k_orb_eval<<<(unsigned)nb, 256, 0, p->stream>>>(a);
    timing_end(p, slot);
    return cuda_check(cudaGetLastError(), "k_orb_eval launch");
}

SL_CHECK_READER(chk_orbital)

}  // namespace sl

extern "C" sl_status sl_quad_factor(double nu_hz, double T0, double *q) {
    if (!q) return sl::set_error(SL_ERR_ARG, "sl_quad_factor: NULL output");
    if (!(nu_hz > 0.0 && nu_hz < HUGE_VAL && T0 > 0.0 && T0 < HUGE_VAL))
        return sl::set_error(SL_ERR_ARG, "sl_quad_factor: nu=%g and T0=%g must be finite and > 0", nu_hz, T0);
    const double h = 6.62607015e-34, kb = 1.380649e-23;   // exact SI values
    const double a = h * nu_hz / (kb * T0);
    *q = 0.5 * a * (std::exp(a) + 1.0) / std::expm1(a);
    return SL_OK;
}
