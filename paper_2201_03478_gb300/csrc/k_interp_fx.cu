// k_interp_fx.cu -- step 2 of the two-step algorithm (Sect. 2.1) for the plans
// with a double-precision cube (SL_FP64, SL_DF64), its sums on the tensor cores:
//
//   c = Re S_0 + 2 sum_{k>=1} Re(e^{ik psi} S_k),   S_k = sum_q w_q F_k(node q)
//
// for the samples of one cell is the small matrix product
//
//   D[q][s] = F_0(q) / 2 + sum_{k>=1} (Re F_k(q) cos(k psi_s) - Im F_k(q) sin(k psi_s)),
//   c_s = 2 sum_q w_q(s) D[q][s],      q = 0 .. p^2 - 1,
//
// over 2 K terms.  At 1/64 of the FP32 rate the FP64 pipe bound the direct form
// (k_interp_f64, one thread per sample: 594 FP64 operations a sample at p = 4,
// K = 16, 0.96 of the measured FP64 peak).  Here both factors are split into six
// FP16 digits (fxdigits.cuh) and 27 digit products run as mma.sync m16n8k16: 16 nodes x 8
// samples of the cell x 8 orders k, exact in the FP32 accumulators, recombined as 64-bit
// integers and weighted with rounding to nearest, so the sum carries the rounding of its
// operands -- 2^-55 of the power of two above the cell's largest |F| (digits of twice the
// range), 2^-54 of |e^{ik psi}| = 1 -- and the products of their low halves, left out.
// Relative L2 error of a TOD against long double, direct sum -> here: LFI-like sky and
// sidelobe beam, K = 16 2.9e-16 -> 1.3e-16 (scan), K = 32 4.3e-16 -> 1.8e-16, p = 6, K = 8
// 3.4e-16 -> 1.9e-16, p = 2 2.4e-16 -> 1.0e-16.  A tile of 16 nodes is exactly the 4 x 4 stencil; the 128-row
// tiles of tcgen05 would be 7/8 padding here, and at 54 MMAs of 2.15 clocks (the
// rate mma.sync measured: 1024 multiply-adds per clock and SM) per 8 samples the
// tensor pipe is not what binds.
//
// One warp walks a stretch of the sorted samples in batches of 32:
//   1. lane per sample: Lagrange weights in FP64, z = e^{i psi} in fixed point
//      (fx_sincos); z^-3 .. z^4 and the weights go to the warp's shared memory;
//   2. per run of samples of one cell: the A operand, digits of F at the p x p nodes
//      relative to the largest |F| of the cell, kept in registers while the cell
//      stays the same (also across batches); the next cell's nodes are on their way
//      to shared memory (cp.async) while the current one's samples are summed;
//   3. per 8 samples of the run: the B operand, each of a quad's four lanes
//      stepping its own orders k = q + 1 + 4 t by X_{t+1} = 2 cos(4 psi) X_t - X_{t-1};
//      27 MMAs per 8 orders; recombination and the weighted sum over the nodes in
//      integers, reduced over the warp by shuffles.
// Every step is exact or rounds per sample, so a sample's value does not depend on
// which others it is called with, as long as the call takes these sums (interp_route).
// Beyond 16 orders the whole of 2 and 3 repeats per 16 orders ("block"), the phases
// advanced by z^16 between them (that keeps every accumulator below 2^24).
// p = 6 has 36 nodes: three row tiles, one after another; p = 2 uses 4 rows of one.
//
// Cells with a non-finite |F| or one outside 2^-959 .. 2^1000, and samples with a
// non-finite psi or weights too large for the fixed-point range (rings spaced very
// unevenly), are evaluated by the direct FP64 sum instead (interp_one_f64).
#include <algorithm>

#include "fxdigits.cuh"
#include "fxweights.cuh"
#include "interp_f64.cuh"
#include "mbar.cuh"
#include "sl_internal.cuh"

namespace sl {

constexpr int kFxWarps = 8;        // warps per CTA, two CTAs per SM
constexpr int kFxStride = 40;      // 64-bit values per row of a warp's shared tables: the 8 x 4
                                   // lanes of a B fragment read 4 rows at 8 columns in 2 wavefronts
template <int P, bool MB>
struct FxRows {
    // rows: (cos, -sin) of exponents -3 .. 4; wt[P]; wp[P]; result; beyond 16 orders also
    // cos(4 psi) and (cos, -sin)(16 psi)
    static constexpr int kWt = 16, kWp = 16 + P, kT = 16 + 2 * P, kC4 = MB ? 17 + 2 * P : 14, kZ16 = 18 + 2 * P;
    static constexpr int kN = (MB ? 20 : 17) + 2 * P;
    // per warp: the rows, then the nodes of one cell as each lane's 2 x 5 values
    static constexpr int kWarp = kN * kFxStride * (int)sizeof(long long) + 10 * 32 * (int)sizeof(double2);
    static constexpr size_t bytes = 256 * sizeof(longlong2) + (size_t)kFxWarps * kWarp;
};

// element offset of stencil node q of cell (i, j): ghost rows read their ring at phi + pi
template <int P>
__device__ __forceinline__ int fx_node(const InterpGeom &g, int i, int j, int q) {
    const int row = i - P / 2 + 1 + q / P;
    int col = j - P / 2 + 1 + q % P, ring = row;
    if (row < 0 || row >= g.R) {
        ring = (row < 0) ? -1 - row : 2 * g.R - 1 - row;
        col += g.nphi >> 1;
    }
    col = (col < 0) ? col + g.nphi : (col >= g.nphi ? col - g.nphi : col);
    if (!SL_GUARD(ring >= 0 && ring < g.R && col >= 0 && col < g.nphi, 0x211u)) return 0;
    return (ring * g.nphi + col) * (g.K + 1);
}

// Exponent field of a cell's scale 2^e, e = field - 1022, from the largest high word: F 2^(63 - e) has to
// leave its digits' biases room, so the next exponent from (1 - 2^-9) 2^e on.
__device__ __forceinline__ int fx_scale_field(uint32_t mx) { return (int)((mx + 0x1000u) >> 20); }

// the direct sum of one sample, out of line (rare)
template <int P>
__device__ __noinline__ double interp_direct(const InterpGeom &g, const double2 *maps, const StencilRec64 *r,
                                             const double *psi) {
    return interp_one_f64<P>(g, maps, *r, *psi);
}

// Tables of one sample, in the rows of its column: weights, z powers, a zero result.  True
// if the sample needs the direct sum: a non-finite psi, or weights out of range.
template <int P, bool MB>
__device__ __forceinline__ bool fx_setup(const InterpGeom &g, const StencilRec64 &r, double ps, const longlong2 *ptab,
                                         long long *col) {
    using Rows = FxRows<P, MB>;
    bool direct = false;
    long long zc, zs;
    double wt[P], wp[P];
    fx_weights<P>(g, (int)(r.cell >> 16) - 1, r.dth, r.fph, wt, wp);
    if (!fx_sincos(ps, ptab, zc, zs)) {             // |psi| >= 2^9 or not finite
        double sp, cp;
        sincos(ps, &sp, &cp);
        direct |= !fx_q62(cp, zc);
        direct |= !fx_q62(sp, zs);
    }
    zs = -zs;
    unsigned long long wsum = 0;                    // sum of |wt| in Q60
#pragma unroll
    for (int a = 0; a < P; ++a) {
        long long v = 0, u = 0;
        direct |= !fx_q62(wt[a], v);
        wsum += (unsigned long long)llabs(v) >> 2;
        col[(Rows::kWt + a) * kFxStride] = v;
        direct |= !fx_q62(wp[a], u);
        col[(Rows::kWp + a) * kFxStride] = u;
    }
    direct |= wsum >= (2ull << 60);                 // keeps the weighted sum below 2^63
    // (cos, -sin) of exponents -3 .. 4
    const long long c2 = fx_mul(zc, zc) - fx_mul(zs, zs), s2 = fx_mul(zc, zs) * 2;
    const long long c3 = fx_mul(c2, zc) - fx_mul(s2, zs), s3 = fx_mul(c2, zs) + fx_mul(s2, zc);
    const long long c4 = fx_mul(c2, c2) - fx_mul(s2, s2), s4 = fx_mul(c2, s2) * 2;
    const long long cs[4] = {kFxOne, zc, c2, c3}, ss[4] = {0, zs, s2, s3};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        col[(2 * (3 - e)) * kFxStride] = cs[e];
        col[(2 * (3 - e) + 1) * kFxStride] = -ss[e];
        if (e > 0) {
            col[(2 * (3 + e)) * kFxStride] = cs[e];
            col[(2 * (3 + e) + 1) * kFxStride] = ss[e];
        }
    }
    col[14 * kFxStride] = c4;
    col[15 * kFxStride] = s4;
    if (MB) col[Rows::kC4 * kFxStride] = c4;
    col[Rows::kT * kFxStride] = 0;
    if (MB) {
        const long long c8 = fx_mul(c4, c4) - fx_mul(s4, s4), s8 = fx_mul(c4, s4) * 2;
        col[Rows::kZ16 * kFxStride] = fx_mul(c8, c8) - fx_mul(s8, s8);
        col[(Rows::kZ16 + 1) * kFxStride] = fx_mul(c8, s8) * 2;
    }
    return direct;
}
// the z powers of the column times z^16
template <int P>
__device__ __forceinline__ void fx_next_block(long long *col) {
    using Rows = FxRows<P, true>;
    const long long z16c = col[Rows::kZ16 * kFxStride], z16s = col[(Rows::kZ16 + 1) * kFxStride];
#pragma unroll 1
    for (int e = 0; e < 8; ++e) {
        const long long c = col[2 * e * kFxStride], v = col[(2 * e + 1) * kFxStride];
        col[2 * e * kFxStride] = fx_mul(c, z16c) - fx_mul(v, z16s);
        col[(2 * e + 1) * kFxStride] = fx_mul(c, z16s) + fx_mul(v, z16c);
    }
}

// This lane's phases of one sample: (cos, -sin)(k psi), k = 16 blk + q4 + 1, + 4, ...
struct FxPhase {
    long long c, s, pc, ps, c4;
    __device__ __forceinline__ FxPhase(const long long *tab, int row_c4, int q4, int col) {
        c = tab[2 * (q4 + 4) * kFxStride + col];
        s = tab[(2 * (q4 + 4) + 1) * kFxStride + col];
        pc = tab[2 * q4 * kFxStride + col];
        ps = tab[(2 * q4 + 1) * kFxStride + col];
        c4 = tab[row_c4 * kFxStride + col];
    }
    __device__ __forceinline__ void step() {
        const long long nc = fx_cheb(c4, c, pc), ns = fx_cheb(c4, s, ps);
        pc = c;
        ps = s;
        c = nc;
        s = ns;
    }
};

// D times the weights of node q for the sample in column sc; at p = 4 both nodes of a lane
// lie in column gr & 3, whose phi weight fx_reduce applies.  |D| < 23.2 x 2^58 and sum |w| < 2 x 1.6
// leave the sums, in units of 2^-56, below 2^63.
template <int P>
__device__ __forceinline__ long long fx_weigh(long long D, const long long *tab, int q, int sc) {
    long long w = tab[(FxRows<P, false>::kWt + q / P) * kFxStride + sc];
    if (P != 4) w = fx_mul_rn(w, tab[(FxRows<P, false>::kWp + q % P) * kFxStride + sc]);
    return fx_mulhi_rn(D, w);
}
// sum over the 8 row groups: `mine` is this lane's part of the sample in column sc, `other`
// its part of the sample that the lane 16 apart goes on with
template <int P>
__device__ __forceinline__ long long fx_reduce(long long mine, long long other, const long long *tab, int gr, int sc) {
    mine += __shfl_xor_sync(0xffffffffu, other, 16);
    if (P == 4) mine = fx_mul_rn(mine, tab[(FxRows<P, false>::kWp + (gr & 3)) * kFxStride + sc]);
    mine += __shfl_xor_sync(0xffffffffu, mine, 8);
    mine += __shfl_xor_sync(0xffffffffu, mine, 4);
    return mine;
}

// Copies this lane's share of the cell's row tile t and block blk into raw: nodes gr and
// gr + 8 of the tile, per node F_0 and the orders 16 blk + q4 + 1 + 4 e (absent ones: zeros).
template <int P>
__device__ __forceinline__ void fx_fetch(const InterpGeom &g, const double2 *__restrict__ maps, unsigned cell, int t,
                                         int blk, int gr, int q4, int lane, double2 *raw) {
    const int i = (int)(cell >> 16) - 1, j = (int)(cell & 0xffffu);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int q = 16 * t + gr + 8 * h;
        if (P * P <= 8 && h == 1) break;
        const bool ok = q < P * P;
        const double2 *src = maps + fx_node<P>(g, i, j, ok ? q : 0);
        cp_async16z(raw + (5 * h) * 32 + lane, src, ok);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = 16 * blk + q4 + 1 + 4 * e;
            cp_async16z(raw + (5 * h + 1 + e) * 32 + lane, src + (k <= g.K ? k : 0), ok && k <= g.K);
        }
    }
    cp_async_commit();
}

// This lane's share of the largest |F| of a cell: high word of the magnitude
template <int P>
__device__ __forceinline__ uint32_t fx_cell_max(const InterpGeom &g, const double2 *__restrict__ maps, unsigned cell, int gr,
                                                int q4) {
    uint32_t mx = 0;
    for (int q = gr; q < P * P; q += 8) {
        const int o = fx_node<P>(g, (int)(cell >> 16) - 1, (int)(cell & 0xffffu), q);
        for (int k = q4; k <= g.K; k += 4) {
            const double2 v = __ldg(maps + o + k);
            // k = 0 enters through its real part only
            mx = max(mx, (uint32_t)__double2hiint(v.x) & 0x7fffffffu);
            if (k > 0) mx = max(mx, (uint32_t)__double2hiint(v.y) & 0x7fffffffu);
        }
    }
    return mx;
}

// Whether this lane's share of a cell holds a value other than zero (k = 0 through its real part).
// Out of line: rare.
__device__ __forceinline__ uint32_t fx_bits(double x) { return ((uint32_t)__double2hiint(x) & 0x7fffffffu) | (uint32_t)__double2loint(x); }
template <int P>
__device__ __noinline__ bool fx_cell_any(const InterpGeom &g, const double2 *__restrict__ maps, unsigned cell, int gr, int q4) {
    uint32_t any = 0;
    for (int q = gr; q < P * P; q += 8) {
        const double2 *v = maps + fx_node<P>(g, (int)(cell >> 16) - 1, (int)(cell & 0xffffu), q);
#pragma unroll 4
        for (int k = q4; k <= g.K; k += 4) {
            const double2 d = __ldg(v + k);
            any |= fx_bits(d.x) | (k > 0 ? fx_bits(d.y) : 0u);
        }
    }
    return any != 0;
}
// The exponent field of a cell's scale; 2047: direct evaluation.  A cell of zeros (a masked region,
// the first step of a fit from zero; any() tells) takes the smallest scale: summed directly, a cube
// of zeros took 23.9 ms for 2e7 samples at K = 16, 1024 x 2048 cells, 11.5 otherwise.
template <typename F>
__device__ __forceinline__ int fx_scale(uint32_t mx, F any) {
    const int ef = fx_scale_field(mx);
    if (ef < 64) return __any_sync(0xffffffffu, any()) ? 2047 : 64;
    return ef > 2022 ? 2047 : ef;
}

// MB: more than 16 orders (several blocks)
template <int P, bool MB>
__global__ void __launch_bounds__(32 * kFxWarps, 2) k_interp_fx(const __grid_constant__ InterpGeom g,
                                                                const double2 *__restrict__ maps,
                                                                const StencilRec64 *__restrict__ rec,
                                                                const double *__restrict__ psi,
                                                                const unsigned *__restrict__ perm, int64_t n, int chunk,
                                                                const unsigned *__restrict__ occ, float min_mean,
                                                                double *__restrict__ tod) {
    constexpr int NQ = P * P, NT = (NQ + 15) / 16, NH = NQ > 8 ? 2 : 1;
    constexpr bool kOne = NT == 1 && !MB;           // one operand per cell: kept across batches, prefetched
    // orders of the digit products kept; without the short form's halves to match, order 6 whole and no 7
    constexpr int NS = P == 4 && !MB ? kFxSums : kFxSums - 1;
    using Rows = FxRows<P, MB>;
    if (occ && (float)n < min_mean * (float)*occ) return;   // few samples per cell: another kernel runs instead
    extern __shared__ __align__(16) unsigned char fx_smem[];
    longlong2 *ptab = reinterpret_cast<longlong2 *>(fx_smem);       // (cos, sin)(2 pi i / 256), Q62
    for (int q = threadIdx.x; q < 256; q += 32 * kFxWarps) ptab[q] = __ldg(g.phase_tab + q);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long *tab = reinterpret_cast<long long *>(fx_smem + 256 * sizeof(longlong2) + (size_t)warp * Rows::kWarp);
    double2 *raw = reinterpret_cast<double2 *>(tab + Rows::kN * kFxStride);     // [2][F_0, 4 orders][32 lanes]
    const int gr = lane >> 2, q4 = lane & 3;        // fragment row group and quad lane
    const int K = g.K;
    const int nblk = MB ? (K + 15) >> 4 : 1;        // blocks of 16 orders
    const int tsh = MB ? 32 - __clz(nblk - 1) : 0;  // headroom of the result's sum over the blocks

    // A operand of the current (cell, row tile, block): digits of nodes gr and gr + 8, orders
    // 16 blk + q4 + 1 + 4 e, e = 0..3, and F_0 / 2 of both nodes
    uint32_t adig[2][kFxDig][4];
    long long f0[2] = {0, 0};
    unsigned a_cell = 0xffffffffu;                  // cell whose operand (kOne) or scale is held
    int a_ef = 0;                                   // its exponent field (2047: direct evaluation)

    const int64_t wfirst = ((int64_t)blockIdx.x * kFxWarps + warp) * chunk;
    const int64_t wlast = min(n, wfirst + chunk);
    if (wfirst >= wlast) return;
    // the batch's sample, record and psi (lanes past the end repeat the last sample), one batch ahead
    unsigned s_next = perm[min(wfirst + lane, wlast - 1)];
    StencilRec64 r_next = rec[s_next];
    double ps_next = psi[s_next];
    if (kOne) fx_fetch<P>(g, maps, __shfl_sync(0xffffffffu, r_next.cell, 0), 0, 0, gr, q4, lane, raw);
    for (int64_t t0 = wfirst; t0 < wlast; t0 += 32) {
        const int cnt = (int)min((int64_t)32, wlast - t0);
        // ---- 1: one sample per lane
        const unsigned s = s_next, mycell = r_next.cell;
        bool direct = fx_setup<P, MB>(g, r_next, ps_next, ptab, tab + lane);     // this sample needs the direct sum
        if (t0 + 32 < wlast) {
            s_next = perm[min(t0 + 32 + lane, wlast - 1)];
            r_next = rec[s_next];
            ps_next = psi[s_next];
        }
        int efs = 0;                                // exponent field of this sample's cell
        const unsigned prev = __shfl_up_sync(0xffffffffu, mycell, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane < cnt && (lane == 0 || mycell != prev));
        __syncwarp();

#pragma unroll 1
        for (int blk = 0; blk < nblk; ++blk) {
            if (MB && blk > 0) {                    // phases of the next 16 orders: times z^16
                __syncwarp();
                fx_next_block<P>(tab + lane);
                __syncwarp();
            }
            // ---- 2: runs of equal cells, [r0, r1)
#pragma unroll 1
            for (int r0 = 0, r1; r0 < cnt; r0 = r1) {
                const unsigned cell = __shfl_sync(0xffffffffu, mycell, r0);
                const unsigned later = r0 < 31 ? heads & (0xfffffffeu << r0) : 0u;
                r1 = later ? __ffs(later) - 1 : cnt;
#pragma unroll 1
                for (int t = 0; t < NT; ++t) {
                    if (cell != a_cell || !kOne) {
                        if (!kOne) fx_fetch<P>(g, maps, cell, t, blk, gr, q4, lane, raw);
                        uint32_t mx = 0;
                        if (!kOne && cell != a_cell)        // the scale needs every row tile and block
                            mx = fx_cell_max<P>(g, maps, cell, gr, q4);
                        cp_async_wait_all();                // each lane reads what it fetched itself
                        if (kOne) {
#pragma unroll
                            for (int v = 0; v < 5 * NH; ++v) {
                                const double2 d = raw[v * 32 + lane];
                                mx = max(mx, (uint32_t)__double2hiint(d.x) & 0x7fffffffu);
                                if (v % 5) mx = max(mx, (uint32_t)__double2hiint(d.y) & 0x7fffffffu);
                            }
                        }
                        if (cell != a_cell) {       // largest exponent over nodes and orders
                            mx = __reduce_max_sync(0xffffffffu, mx);
                            a_ef = fx_scale(mx, [&] { return fx_cell_any<P>(g, maps, cell, gr, q4); });
                            a_cell = cell;
                        }
                        if (a_ef < 2047) {
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (h >= NH) {
#pragma unroll
                                    for (int e = 0; e < 4; ++e)
#pragma unroll
                                        for (int u = 0; u < kFxDig; ++u) adig[e >> 1][u][2 * (e & 1) + h] = 0;
                                    continue;
                                }
                                // ghost rows flip the odd orders k = q4 + 1 + 4 e of this lane
                                const int row = (int)(cell >> 16) - P / 2 + (16 * t + gr + 8 * h) / P;
                                const bool flip = (row < 0 || row >= g.R) && !(q4 & 1);
                                f0[h] = blk == 0 ? fx_from_double(raw[(5 * h) * 32 + lane].x, a_ef) >> 5 : 0;
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    uint32_t d[kFxDig] = {0, 0, 0, 0, 0, 0};
                                    if (4 * e < K - 16 * blk) {
                                        const double2 v = raw[(5 * h + 1 + e) * 32 + lane];
                                        long long x = fx_from_double<63>(v.x, a_ef), y = fx_from_double<63>(v.y, a_ef);
                                        if (flip) { x = -x; y = -y; }
                                        fx_digits<true>(x, y, d);
                                    }
#pragma unroll
                                    for (int u = 0; u < kFxDig; ++u) adig[e >> 1][u][2 * (e & 1) + h] = d[u];
                                }
                            }
                        }
                    }
                    if (kOne) {                     // the stretch's next cell, at one place (code size)
                        const unsigned here = __shfl_sync(0xffffffffu, mycell, r1 & 31);
                        const unsigned ahead = __shfl_sync(0xffffffffu, r_next.cell, 0);
                        if (r1 < cnt || (t0 + 32 < wlast && ahead != cell))
                            fx_fetch<P>(g, maps, r1 < cnt ? here : ahead, 0, 0, gr, q4, lane, raw);
                    }
                    const bool mine_in_run = lane >= r0 && lane < r1;
                    if (a_ef == 2047) {             // uniform over the warp: no row tile is summed
                        direct |= mine_in_run;
                        break;
                    }
                    if (mine_in_run) efs = a_ef;
                    // ---- 3: groups of 8 samples
#pragma unroll 1
                    for (int c0 = r0; c0 < r1; c0 += 8) {
                        float acc[4][NS];           // [node h, sample e as 2 h + e][s]
                        FxPhase ph(tab, Rows::kC4, q4, min(c0 + gr, 31));   // past the run: a column of no use
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            if (b == 0 || 16 * blk + 8 < K) {      // K = 0: both operands are zero digits
                                uint32_t b0[kFxDig], b1[kFxDig] = {0, 0, 0, 0, 0, 0};
                                fx_digits(ph.c, ph.s, b0);
                                ph.step();
                                if (16 * blk + 8 * b + 4 < K) fx_digits(ph.c, ph.s, b1);
                                if (b == 0) ph.step();
#pragma unroll
                                for (int u = 0; u < kFxDig; ++u)
#pragma unroll
                                    for (int v = 0; v < kFxDig; ++v)
                                        if (NS == kFxSums ? u < 3 || v < 3 : u + v < NS)
                                            mma_f16(acc[0][u + v], acc[1][u + v], acc[2][u + v], acc[3][u + v], adig[b][u],
                                                    b0[v], b1[v], b == 0 && (u == 0 || (u < 3 && v == 5)));
                            }
                        }
                        // weighted sum over this lane's two nodes, samples c0 + 2 q4 + {0, 1}
                        long long T[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            T[e] = 0;
#pragma unroll
                            for (int h = 0; h < NH; ++h) {
                                const int q = 16 * t + gr + 8 * h;
                                if (NQ >= 16 * (t + 1) || q < NQ)
                                    T[e] += fx_weigh<P>(fx_combine(acc[2 * h + e]) + f0[h], tab, q, min(c0 + 2 * q4 + e, 31));
                            }
                        }
                        // lanes with gr < 4 go on with the even sample
                        const int sc = c0 + 2 * q4 + (gr >> 2);
                        const long long mine = fx_reduce<P>((gr < 4) ? T[0] : T[1], (gr < 4) ? T[1] : T[0], tab, gr, min(sc, 31));
                        if ((gr & 3) == 0 && sc < r1) tab[Rows::kT * kFxStride + sc] += fx_shift_even(mine, tsh);
                    }
                }
            }
        }
        __syncwarp();
        if (lane < cnt) {
            double out;
            if (direct) {
                out = interp_direct<P>(g, maps, rec + s, psi + s);
            } else {
                // c = 2 T 2^-56 2^e, e = ef - 1022
                const double sc = __longlong_as_double((long long)(efs - 54 + tsh) << 52);
                out = (double)tab[Rows::kT * kFxStride + lane] * sc;
            }
            tod[s] = out;
        }
        __syncwarp();
    }
    cp_async_wait_all();
}

// ------------------------------------------------------------------ few samples per cell
// The same sums on the integer pipe, for sorts that leave few samples per occupied cell:
// there the columns of k_interp_fx's products would be mostly empty.  One warp per batch
// of 32 samples as there, the phases split into halves per lane beforehand; then sample by
// sample, each lane 2 nodes x 4 orders: F as (xh, xl), kept while the cell stays the same,
// three multiply-adds per real term, sums over the quad by shuffles, weights as there.
// NE blocks of four orders: with fewer, more warps fit (4 CTAs an SM up to 8 orders, 3 above:
// 403 -> 319 us at K = 4, 1e6 samples in as many cells); small calls take fewer samples a warp.
// The next cell's nodes are loaded while the current sample is summed.  Bound by the
// integer pipe (20 instructions per real value of F); the cube is read in 64-byte pieces
// per quad, where one sample per thread reads 16-byte pieces from 32 lines at a time and
// waits for the L1 tags (2.1 ms at K = 16 and 1e6 samples in as many cells).  Every value
// is that of k_interp_fx, bit for bit.
constexpr int kFxsWarps = 4;
constexpr int kFxsPhStride = 33;   // 16-byte entries per order: a quad's 4 orders in distinct banks

template <int NE>
__global__ void __launch_bounds__(32 * kFxsWarps, NE <= 2 ? 4 : 3) k_interp_fx_short(const __grid_constant__ InterpGeom g,
                                                                       const double2 *__restrict__ maps,
                                                                       const StencilRec64 *__restrict__ rec,
                                                                       const double *__restrict__ psi,
                                                                       const unsigned *__restrict__ perm, int64_t n, int bs,
                                                                       const unsigned *__restrict__ occ, float min_mean,
                                                                       double *__restrict__ tod) {
    if (!((float)n < min_mean * (float)*occ)) return;       // k_interp_fx runs instead
    constexpr int P = 4;
    using Rows = FxRows<P, false>;
    extern __shared__ __align__(16) unsigned char fx_smem[];
    longlong2 *ptab = reinterpret_cast<longlong2 *>(fx_smem);
    for (int q = threadIdx.x; q < 256; q += 32 * kFxsWarps) ptab[q] = __ldg(g.phase_tab + q);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int4 *ph = reinterpret_cast<int4 *>(fx_smem + 256 * sizeof(longlong2)) + (size_t)warp * 4 * NE * kFxsPhStride;
    long long *tab = reinterpret_cast<long long *>(fx_smem + 256 * sizeof(longlong2) +
                                                   (size_t)kFxsWarps * 4 * NE * kFxsPhStride * sizeof(int4)) +
                     (size_t)warp * Rows::kN * kFxStride;
    const int gr = lane >> 2, q4 = lane & 3;
    const int K = g.K;
    const int64_t nbatch = (n + bs - 1) / bs;
    for (int64_t batch = (int64_t)blockIdx.x * kFxsWarps + warp; batch < nbatch; batch += (int64_t)gridDim.x * kFxsWarps) {
        const int64_t t0 = batch * bs;
        const int cnt = (int)min((int64_t)bs, n - t0);
        const unsigned s = perm[t0 + min(lane, cnt - 1)];
        unsigned mycell;
        bool direct;
        {
            const StencilRec64 r = rec[s];
            mycell = r.cell;
            direct = fx_setup<P, false>(g, r, psi[s], ptab, tab + lane);
        }
        int efs = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            FxPhase f(tab + lane, Rows::kC4, q, 0);
#pragma unroll 1
            for (int e = 0; e < NE && 4 * e + q < K; ++e) {
                int4 v;
                fx_split(f.c, v.x, v.y);
                fx_split(f.s, v.z, v.w);
                ph[(4 * e + q) * kFxsPhStride + lane] = v;
                f.step();
            }
        }
        __syncwarp();
        unsigned a_cell = 0xffffffffu;
        int a_ef = 0;
        int ah[2][NE][2], al[2][NE][2];
        long long f0[2] = {0, 0};
        double2 raw[2][NE];
        double raw0[2];
        auto fetch = [&](unsigned cell) {
            const int i = (int)(cell >> 16) - 1, j = (int)(cell & 0xffffu);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const double2 *src = maps + fx_node<P>(g, i, j, gr + 8 * h);
                raw0[h] = __ldg(&src->x);
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    const int k = q4 + 1 + 4 * e;
                    raw[h][e] = k <= K ? __ldg(src + k) : make_double2(0.0, 0.0);
                }
            }
        };
        fetch(__shfl_sync(0xffffffffu, mycell, 0));
#pragma unroll 1
        for (int c = 0; c < cnt; ++c) {
            const unsigned cell = __shfl_sync(0xffffffffu, mycell, c);
            if (cell != a_cell) {
                uint32_t mx = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mx = max(mx, (uint32_t)__double2hiint(raw0[h]) & 0x7fffffffu);
#pragma unroll
                    for (int e = 0; e < NE; ++e)
                        mx = max(mx, max((uint32_t)__double2hiint(raw[h][e].x) & 0x7fffffffu,
                                         (uint32_t)__double2hiint(raw[h][e].y) & 0x7fffffffu));
                }
                mx = __reduce_max_sync(0xffffffffu, mx);
                a_ef = fx_scale(mx, [&] { return fx_cell_any<P>(g, maps, cell, gr, q4); });
                a_cell = cell;
                if (a_ef < 2047) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int row = (int)(cell >> 16) - P / 2 + (gr + 8 * h) / P;
                        const bool flip = (row < 0 || row >= g.R) && !(q4 & 1);
                        f0[h] = fx_from_double(raw0[h], a_ef) >> 5;
#pragma unroll
                        for (int e = 0; e < NE; ++e) {
                            if (4 * e >= K) continue;
                            long long x = fx_from_double<63>(raw[h][e].x, a_ef), y = fx_from_double<63>(raw[h][e].y, a_ef);
                            if (flip) { x = -x; y = -y; }
                            fx_split<true>(x, ah[h][e][0], al[h][e][0]);
                            fx_split<true>(y, ah[h][e][1], al[h][e][1]);
                        }
                    }
                }
                // the next cell of the batch
                const unsigned after = __ballot_sync(0xffffffffu, mycell != cell && lane > c && lane < cnt);
                if (after) fetch(__shfl_sync(0xffffffffu, mycell, __ffs(after) - 1));
            }
            if (lane == c) {
                efs = a_ef;
                direct |= a_ef == 2047;
            }
            if (a_ef == 2047) continue;
            long long hh[2] = {0, 0}, xx[2] = {0, 0};
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                if (4 * e >= K) continue;
                // orders past K: F is zero there, and so is the product with whatever ph holds
                const int4 y = ph[(4 * e + q4) * kFxsPhStride + c];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    hh[h] += (long long)ah[h][e][0] * y.x;
                    hh[h] += (long long)ah[h][e][1] * y.z;
                    xx[h] += (long long)ah[h][e][0] * y.y;
                    xx[h] += (long long)al[h][e][0] * y.x;
                    xx[h] += (long long)ah[h][e][1] * y.w;
                    xx[h] += (long long)al[h][e][1] * y.z;
                }
            }
            // over the quad: lanes with q4 < 2 go on with node gr, the others with gr + 8
            const bool up = q4 >= 2;
            long long H = up ? hh[1] : hh[0], X = up ? xx[1] : xx[0];
            H += __shfl_xor_sync(0xffffffffu, up ? hh[0] : hh[1], 2);
            X += __shfl_xor_sync(0xffffffffu, up ? xx[0] : xx[1], 2);
            H += __shfl_xor_sync(0xffffffffu, H, 1);
            X += __shfl_xor_sync(0xffffffffu, X, 1);
            long long mine = fx_weigh<P>(fx_combine(H, X) + (up ? f0[1] : f0[0]), tab, gr + (up ? 8 : 0), c);
            mine += __shfl_xor_sync(0xffffffffu, mine, 2);
            mine = fx_reduce<P>(mine, mine, tab, gr, c);
            if (lane == 0) tab[Rows::kT * kFxStride + c] = mine;
        }
        __syncwarp();
        if (lane < cnt)
            tod[s] = direct ? interp_direct<P>(g, maps, rec + s, psi + s)
                            : (double)tab[Rows::kT * kFxStride + lane] * __longlong_as_double((long long)(efs - 54) << 52);
        __syncwarp();
    }
}

static size_t fx_short_smem(int ne) {
    return 256 * sizeof(longlong2) + (size_t)kFxsWarps * (4 * ne * kFxsPhStride * sizeof(int4) +
                                                          FxRows<4, false>::kN * kFxStride * sizeof(long long));
}

SL_CHECK_READER(chk_interp_fx)

constexpr int64_t kFxFew = 20480;   // some 8 samples a warp of k_interp_fx

// Which calls take the fixed-point sums (FP64 plans otherwise k_interp_f64, DF64 plans
// k_interp_df).  A cell's operand costs the same at every K, so few orders need many samples per
// cell.  At p = 4 and below 11 orders the line is the density of uniform samples (the slowest form: a
// scan fills fewer cells) at which they break even (time over the direct sum's, FP64, 127 x 128, 256 x
// 512 and 1024 x 2048 cells): K = 1 1.19, 0.86 at 61 and 122 per cell; K = 2 1.19, 0.94 at 37 and
// 61; K = 3 1.26, 0.89 at 6 and 12; K = 4 1.02, 0.84 at 2.3 and 4.6; K = 8 1.14, 0.89 at 0.5 and
// 1.4.  K = 0 gains nothing.  With at most some 8 samples for every warp of the chip (kFxFew), the
// products of a cell take less time than one thread's sums: from 4 orders on 12 against 21 us (1000
// samples); a scan gains to the end of that range, uniform samples even out at 1e4 with K = 4 and 5, 1.4e4
// with 6 and 2e4 with 8 and lose up to 6 us of a call beyond, which stays so that these calls give a
// sample one value whatever their size.
// From 11 orders on the fixed-point sums are always taken.  Sparse uniform samples, nearly every one in
// a cell of its own, lose by it (interp_tod's time over that with the direct sum at 1.12, 1.33 and 1.71 samples
// per occupied cell, 300 x 600 cells: K = 11 1.15, 1.14, 0.97; 12 1.05, 1.10, 0.91; 14 1.09, 1.14, 0.94; 16 1.04, 1.04,
// 0.86; 1024 x 2048: 1.15, 1.07, 0.94; 1.08, 1.00, 0.89; 1.14, 1.06, 0.93; 1.04, 0.96, 0.84), a scan at the same size gains
// up to half (one pointing period, 0.05 per grid cell: 0.53).  Only the sort's count of occupied cells
// tells them apart: a launch of the direct sum beside the others costs every such call 4 us (5% of a
// scan's), and inside k_interp_fx, whose shared memory takes its L1, it is 2 to 3 times slower.
// For p = 2 and 6 and beyond 16 orders there is only the tensor-core
// form, whose operands cost several row tiles or blocks per cell: from 48 samples per grid
// cell on (K = 32, p = 6, 55 per cell: 22 [43] ms; 5.5 per cell: 11 [4.4]; K = 8, p = 2: 1.6 [2.3]
// and 0.60 [0.24]), 96 below 8 orders (K = 4: 1.26 at 61, 0.91 at 122), none below 3 (K = 2: 1.2 at 122).
// DF64's alternative is faster: 13 to 16 orders from 8 samples per grid cell on, and there by the
// occupied cells again, with both forms launched (time of k_interp_fx over the double-float form's, uniform samples
// at 16, 30 and 60 per cell, 300 x 600 cells: K = 13 1.35, 1.22, 0.95; K = 16 1.17, 1.03, 0.79; 1024 x 2048, beyond L2: 0.95,
// 0.94, 0.82; 0.79, 0.80, 0.70, and at 8 1.4 and 1.25; a scan, 200 and more per occupied cell: 0.36-0.70); 8
// orders lose 1.35 at 61 per cell.
// What the host decides, it decides by the whole TOD's samples per grid cell, so that every piece of a
// TOD gets the same kernels.
InterpRoute interp_route(const sl_plan *p, int64_t n_total, float *min_mean) {
    *min_mean = 0.f;
    if (plan_fp32(p->precision)) return InterpRoute::plain;
    const double cells = (double)(p->R + 1) * p->nphi, per_cell = (double)n_total / cells;
    if (p->precision == SL_DF64) {
        if (p->p != 4 || p->K <= 12 || p->K > 16 || per_cell < 8.0) return InterpRoute::plain;
        const bool in_l2 = 16.0 * (double)p->R * p->nphi * (p->K + 1) <= 1e8;       // the cube
        *min_mean = in_l2 ? 56.f - 8.f * (float)(p->K - 13) : 16.f;
        return per_cell >= (double)*min_mean ? InterpRoute::fx : InterpRoute::by_occupancy;     // occupied <= all cells
    }
    if (p->p != 4 || p->K > 16)
        return p->K > 2 && per_cell >= (p->K < 8 ? 96.0 : 48.0) ? InterpRoute::fx : InterpRoute::plain;
    if (p->K >= 4 && n_total <= kFxFew) return InterpRoute::fx;
    constexpr double kLine[11] = {0.0, 96.0, 48.0, 8.0, 4.0, 4.0, 4.0, 4.0, 2.0, 2.0, 2.0};
    return p->K > 10 || (p->K > 0 && per_cell >= kLine[p->K]) ? InterpRoute::fx : InterpRoute::plain;
}

sl_status launch_interp_fx(sl_plan *p, const SortBufs &b, const void *maps, const double *psi, int64_t n, const unsigned *occ,
                           float min_mean, double *tod) {
    void (*kern)(const InterpGeom, const double2 *, const StencilRec64 *, const double *, const unsigned *, int64_t, int,
                 const unsigned *, float, double *) = nullptr;
    const bool mb = p->K > 16;
    size_t sm = 0;
#define SL_FX(PV, MBV)                        \
    if (p->p == PV && mb == MBV) {            \
        kern = k_interp_fx<PV, MBV>;          \
        sm = FxRows<PV, MBV>::bytes;          \
    }
    SL_FX(2, false) SL_FX(2, true) SL_FX(4, false) SL_FX(4, true) SL_FX(6, false) SL_FX(6, true)
#undef SL_FX
    if (!kern) return set_error(SL_ERR_UNSUPPORTED, "interp_order %d", p->p);
    cudaError_t e = allow_dyn_smem(kern, sm);
    if (e != cudaSuccess) return cuda_check(e, "k_interp_fx smem attribute");
    // a warp's stretch: long enough that a cell's operand is rarely built twice (512), short
    // enough that small calls fill the SMs (2 CTAs of 8 warps each; a call of 1000 samples
    // waits for one cell per warp, not for 32 in a row)
    int nsm = 152;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
    const int64_t full = (int64_t)nsm * 2 * kFxWarps;            // warps of one wave
    const int64_t waves = std::max<int64_t>(1, (n + full * 512 - 1) / (full * 512));
    const int64_t per = (n + full * waves - 1) / (full * waves);  // whole waves
    const int chunk = (int)(per <= 32 ? std::max<int64_t>(per, 1) : (per + 31) / 32 * 32);
    // Few samples per occupied cell take less time in k_interp_fx_short (equal at 23: K = 16, 3e6
    // samples on 256 x 512 cells 1.46 and 1.49 ms; at 12, 2e5 on 127 x 128: 0.20 and 0.13 ms; K = 4 at
    // 15, 2e6: 0.87 and 0.66).  When that may be the case and the call is large enough to fill
    // the SMs both are launched, and the sort's count of occupied cells decides on the device
    // which one runs (the other returns at once).
    constexpr float kMean = 24.f;
    const bool both = p->p == 4 && !mb && p->precision != SL_DF64 && n > 4 * full && (float)n < kMean * (float)p->nkeys;
    if (both) {
        const int ne = std::max(1, (p->K + 3) / 4), ctas = nsm * (ne <= 2 ? 4 : 3);
        auto short_kern = ne == 1 ? k_interp_fx_short<1> : ne == 2 ? k_interp_fx_short<2> : ne == 3 ? k_interp_fx_short<3>
                                                                                         : k_interp_fx_short<4>;
        const size_t sm_short = fx_short_smem(ne);
        e = allow_dyn_smem(short_kern, sm_short);
        if (e != cudaSuccess) return cuda_check(e, "k_interp_fx_short smem attribute");
        const int slot = timing_begin(p, "interp_fx_short");
        const int64_t one = (int64_t)ctas * kFxsWarps;              // warps of one wave
        const int64_t bs = std::max<int64_t>(4, std::min<int64_t>(32, (n + one - 1) / one));
        const int64_t nb = (n + bs * kFxsWarps - 1) / (bs * kFxsWarps);
        short_kern<<<(unsigned)std::min<int64_t>(nb, ctas), 32 * kFxsWarps, sm_short, p->stream>>>(
            p->geom, (const double2 *)maps, (const StencilRec64 *)b.rec, psi, b.perm, n, (int)bs, b.occ, kMean, tod);
        timing_end(p, slot);
    }
    const int64_t nwarps = (n + chunk - 1) / chunk;
    const unsigned grid = (unsigned)((nwarps + kFxWarps - 1) / kFxWarps);
    int slot = timing_begin(p, "interp_fx");
    kern<<<grid, 32 * kFxWarps, sm, p->stream>>>(p->geom, (const double2 *)maps, (const StencilRec64 *)b.rec, psi, b.perm, n,
                                                 chunk, both ? b.occ : occ, both ? kMean : min_mean, tod);
    timing_end(p, slot);
    return cuda_check(cudaGetLastError(), "k_interp_fx launch");
}

}  // namespace sl
