// lcontract.cuh -- arguments, block layout and output of the spin "Legendre" step's
// kernels (k_lcontract.cu, k_lcontract_fx.cu).
#pragma once

#include "sl_internal.cuh"

namespace sl {

struct LcArgs {
    int L, K, ncomp, R, npairs, nchunk, ppt;  // ppt: ring pairs per thread
    int64_t nalm;
    const double2 *sky, *beam;       // FP64 inputs
    const float2 *sky32, *beam32;    // FP32 copies (FP32 plans)
    const double *xr;
    const float *y32;
    const int *ls;
    const double2 *st64;
    const float2 *st32;
    const RTab64 *tab64;
    const RTab32 *tab32;
    void *G;
};

// Block b -> (m, k, ring chunk pc).
__device__ __forceinline__ void block_mk_of(const LcArgs &a, int b, int &m, int &k, int &pc) {
    pc = b % a.nchunk;
    b /= a.nchunk;
    k = b % (a.K + 1);
    m = b / (a.K + 1);
}
__device__ __forceinline__ void block_mk(const LcArgs &a, int &m, int &k, int &pc) { block_mk_of(a, blockIdx.x, m, k, pc); }

__device__ __forceinline__ int64_t start_index(const LcArgs &a, int k, int m, int neg, int pair) {
    return (((int64_t)k * (a.L + 1) + m) * 2 + neg) * a.npairs + pair;
}

// Writes one sum of one recurrence.  neg = 0 (+k): sum 0 -> (north, +m), sum 1 ->
// (south, -m); neg = 1 (-k): sum 0 -> (north, -m), sum 1 -> (south, +m).
template <typename C>
__device__ __forceinline__ void write_one(const LcArgs &a, int m, int k, int pair, int neg, int which, C v) {
    C *G = reinterpret_cast<C *>(a.G);
    const int rn = pair, rs = a.R - 1 - pair;
    const bool minus = neg != which;            // row (k, L - m) of G, else (k, L + m)
    if ((minus && m == 0) || (which && rs == rn)) return;
    const bool flip = which ? (neg ? (m & 1) : ((m ^ k) & 1)) : (neg && (k & 1));
    if (flip) { v.x = -v.x; v.y = -v.y; }
    G[((int64_t)k * (2 * a.L + 1) + (minus ? a.L - m : a.L + m)) * a.R + (which ? rs : rn)] = v;
}
template <typename C>
__device__ __forceinline__ void write_two(const LcArgs &a, int m, int k, int pair, int neg, C acc1, C acc2) {
    write_one(a, m, k, pair, neg, 0, acc1);
    write_one(a, m, k, pair, neg, 1, acc2);
}

sl_status launch_lcontract_fx(sl_plan *p, const LcArgs &a);

}  // namespace sl
