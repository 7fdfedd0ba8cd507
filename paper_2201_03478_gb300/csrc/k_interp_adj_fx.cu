// k_interp_adj_fx.cu -- transpose of the interpolation (k_interp.cu: maps_bar_k(node) +=
// w_node y eps_k e^{-ik psi}) in fixed point and on the tensor cores, at p = 4:
//
//   Fbar[q][c] = sum_s (y_s w_q(s)) E_c(s),   q: 16 nodes of the cell, c: (cos, -sin)(k psi_s)
//
// The FP64 form (k_interp_adjoint) was bound by the FP64 pipe: 2 p^2 (K + 1) multiply-adds a
// sample at 1/64 of the FP32 rate.  Here both factors are
// split into FP16 digits (fxdigits.cuh) and summed over 16 samples of a cell per mma.sync
// m16n8k16, exactly; the 16 nodes of a 4 x 4 stencil are the 16 rows of the tile (as in
// k_interp_fx, tcgen05's 128 rows would be mostly padding).
//
// One warp walks a stretch of the sorted samples in batches of 32:
//   1. lane per sample: weights and phases in fixed point (fx_sincos; X_{k+1} = 2 cos psi X_k -
//      X_{k-1}), y w_q relative to the largest |y| of the sample's run of equal cells, as
//      digits to the warp's shared memory, [digit][node or real][sample];
//   2. per 4 orders (their phases' digits made just before) and run: A = the run's columns
//      (the others masked to zero), 27 digit products per 16 samples (order 0: E = 1, six),
//      recombined and added to 64-bit sums in shared memory with an exponent per column.
// The node of row q is kept at slot (column mod 4): when the run moves to a neighbouring cell
// only the columns that leave the stencil are added to the cube (atomically), a quarter of the
// values when the next cell is the next column.
//
// Measured (before -> after): 5e6 scanning samples at K = 16, 1024 x 2048 cells 7.62 -> 1.47 ms;
// 2e7 uniform ones there 28.5 -> 16.0 ms (9.5 a cell); 1e7 at K = 4, 127 x 128 cells 5.21 -> 1.83 ms.
// Bound by issue and the integer pipe (54% and 46% of their rates at 48 samples a cell, K = 16,
// with 2.8 warps a scheduler): digits of 16 nodes and 2 K + 1 phases a sample, recombination a run.
//
// A sample with a non-finite y or psi, |y| outside 2^-959 .. 2^960, or weights out of the
// fixed-point range is scattered in FP64 (adj_one).
#include <algorithm>

#include "fxdigits.cuh"
#include "fxweights.cuh"
#include "interp_f64.cuh"
#include "mbar.cuh"
#include "sl_internal.cuh"

namespace sl {

constexpr int kFaWarps = 4;
constexpr int kFaRow = 16;         // words per row of 32 samples, swizzled (fa_word)
constexpr int kFaDig = 7;          // digits of y w (the phases have six); products of orders 0 to 6
constexpr int kFaEmpty = -4096;    // exponent of sums that are all zero
constexpr int kFaChunk = 512;      // longest stretch of a warp: keeps the 64-bit sums in range

struct FaWarp {                    // one warp's shared memory; sums follow (fa_sums)
    uint32_t a[kFaDig][16][kFaRow];     // digits of y w: [digit][4 row + column mod 4][sample pair]
    uint32_t e[6][8][kFaRow];      // digits of the phases of 4 orders: [digit][2 order + part][sample pair]
};
// Word w of row r: the eight rows and four words of a fragment in distinct banks, without padding
// (rows of 20 words took a fifth more shared memory, and the fourth CTA of an SM up to 8 orders).
__device__ __forceinline__ int fa_word(int r, int w) { return w ^ (((r >> 1) & 3) << 2); }
// bytes per warp with the sums of order 0 (2 rows) and of blocks of 4 orders (2 rows x re, im)
__host__ __device__ __forceinline__ size_t fa_warp_bytes(int nblk) {
    return sizeof(FaWarp) + (size_t)(2 + 4 * nblk) * 32 * sizeof(long long);
}

struct FaArgs {
    InterpGeom g;
    const double *psi, *y;
    const StencilRec64 *rec;
    const unsigned *perm;
    const unsigned *occ;           // with min_mean: run only if n >= min_mean *occ
    float min_mean;
    int64_t n;
    int chunk;
    double2 *fbar;
};

// Cube element of stencil row a's and column col's node (order 0) and whether odd orders flip.
__device__ __forceinline__ int64_t fa_node(const InterpGeom &g, int row, int col, bool &flip) {
    int ring = row;
    flip = row < 0 || row >= g.R;
    if (flip) {
        ring = (row < 0) ? -1 - row : 2 * g.R - 1 - row;
        col += g.nphi >> 1;
    }
    col = (col < 0) ? col + g.nphi : (col >= g.nphi ? col - g.nphi : col);
    if (!SL_GUARD(ring >= 0 && ring < g.R && col >= 0 && col < g.nphi, 0x221u)) return 0;
    return ((int64_t)ring * g.nphi + col) * (g.K + 1);
}

// One sample in FP64 (rare).
__device__ __noinline__ void adj_one(const FaArgs &A, unsigned s) {
    const InterpGeom &g = A.g;
    const StencilRec64 r = A.rec[s];
    const int i = (int)(r.cell >> 16) - 1, j = (int)(r.cell & 0xffffu);
    double wt[4], wp[4], sp, cp;
    weights64<4>(g, i, r.dth, r.fph, wt, wp);
    sincos(A.psi[s], &sp, &cp);
    const double y = A.y[s], c2 = 2.0 * cp;
    for (int q = 0; q < 16; ++q) {
        bool flip;
        double2 *o = A.fbar + fa_node(g, i - 1 + q / 4, j - 1 + q % 4, flip);
        const double w = wt[q / 4] * wp[q % 4];
        double ck = 1.0, sk = 0.0, ckm = cp, skm = -sp;
        for (int k = 0; k <= g.K; ++k) {
            const double f = ((flip && (k & 1)) ? -w : w) * (k ? 2.0 * y : y);
            atomicAdd(&o[k].x, f * ck);
            atomicAdd(&o[k].y, -f * sk);
            const double cn = fma(c2, ck, -ckm), sn = fma(c2, sk, -skm);
            ckm = ck;
            skm = sk;
            ck = cn;
            sk = sn;
        }
    }
}

__global__ void __launch_bounds__(32 * kFaWarps, 4) k_interp_adj_fx(const __grid_constant__ FaArgs A) {
    const InterpGeom &g = A.g;
    if (A.occ && (float)A.n < A.min_mean * (float)*A.occ) return;   // few samples per cell: k_interp_adjoint
    extern __shared__ __align__(16) unsigned char fa_smem[];
    longlong2 *ptab = reinterpret_cast<longlong2 *>(fa_smem);
    for (int q = threadIdx.x; q < 256; q += 32 * kFaWarps) ptab[q] = __ldg(g.phase_tab + q);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gr = lane >> 2, q4 = lane & 3;
    const int nblk = (g.K + 3) >> 2;
    FaWarp &W = *reinterpret_cast<FaWarp *>(fa_smem + 256 * sizeof(longlong2) + (size_t)warp * fa_warp_bytes(nblk));
    // this lane's sums, times 2^(54 - exponent): order 0 of rows gr and gr + 8 (lanes q4 = 0), then
    // per block b re and im of order 1 + 4 b + q4 of both rows
    long long *sums = reinterpret_cast<long long *>(&W + 1) + lane;
    const int64_t wfirst = ((int64_t)blockIdx.x * kFaWarps + warp) * A.chunk, wlast = min(A.n, wfirst + A.chunk);
    if (wfirst >= wlast) return;
    for (int v = 0; v < 2 + 4 * nblk; ++v) sums[32 * v] = 0;
    int ecur = kFaEmpty;                            // exponent of this lane's column's sums
    unsigned cur = 0xffffffffu;                     // the cell whose stencil the sums belong to

    // adds the columns [c_lo, c_hi) (at most four, those of cell c) of block b (-1: order 0) to the cube
    auto flush = [&](int b, unsigned c, int &e, int c_lo, int c_hi) {
        const int i = (int)(c >> 16) - 1;
        // this lane's rows both lie in slot gr & 3: the stencil column with that residue
        const int col = c_lo + ((gr - c_lo) & 3);
        if (col >= c_hi || e == kFaEmpty) return;
        const double sc = __longlong_as_double((long long)(1023 + e - 54) << 52);
        const int k = 1 + 4 * b + q4;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bool flip;
            double2 *o = A.fbar + fa_node(g, i - 1 + (gr >> 2) + 2 * h, col, flip);
            if (b < 0) {
                if (q4 == 0 && sums[32 * h]) atomicAdd(&o[0].x, (double)sums[32 * h] * sc);
                sums[32 * h] = 0;
            } else {
                long long *v = sums + 32 * (2 + 4 * b + 2 * h);
                const double s2 = (flip && (k & 1)) ? -2.0 * sc : 2.0 * sc;    // eps_k = 2, (-1)^k
                if (k <= g.K) {
                    atomicAdd(&o[k].x, (double)v[0] * s2);
                    atomicAdd(&o[k].y, (double)v[32] * s2);
                }
                v[0] = v[32] = 0;
            }
        }
        e = kFaEmpty;
    };

    unsigned s_next = A.perm[min(wfirst + lane, wlast - 1)];
    StencilRec64 r_next = A.rec[s_next];
    double ps_next = A.psi[s_next], y_next = A.y[s_next];
    for (int64_t t0 = wfirst; t0 < wlast; t0 += 32) {
        const int cnt = (int)min((int64_t)32, wlast - t0);
        // ---- 1: one sample per lane
        const unsigned s = s_next, mycell = r_next.cell;
        const unsigned prev = __shfl_up_sync(0xffffffffu, mycell, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane < cnt && (lane == 0 || mycell != prev));
        int ey;                                     // exponent field of the largest |y| of this sample's run
        long long zc, zs;
        {
            double wt[4], wp[4];
            const int i = (int)(mycell >> 16) - 1, j = (int)(mycell & 0xffffu);
            fx_weights<4>(g, i, r_next.dth, r_next.fph, wt, wp);
            long long lwt[4], lwp[4];
            const double y = y_next;
            const int yf = (__double2hiint(y) >> 20) & 0x7ff;
            bool ok = fx_sincos(ps_next, ptab, zc, zs);
            if (!ok) {                              // |psi| >= 2^9 or not finite
                double sp, cp;
                sincos(ps_next, &sp, &cp);
                ok = fx_q62(cp, zc) && fx_q62(sp, zs);
            }
            unsigned long long wsum = 0;            // sum of |wt| in Q60
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                lwt[a] = lwp[a] = 0;
                ok = fx_q62(wt[a], lwt[a]) && ok;
                ok = fx_q62(wp[a], lwp[a]) && ok;
                wsum += (unsigned long long)llabs(lwt[a]) >> 2;
            }
            // sum |wt| < 1.5 (1.25 on uniform rings): |wt| < 1.25, so that 512 samples' sums stay
            // below 2^63
            ok = ok && wsum < (3ull << 59) && (y == 0.0 || (yf >= 64 && yf <= 1983));
            if (!ok && lane < cnt) adj_one(A, s);
            const bool use = ok && lane < cnt && y != 0.0;
            // the run's largest exponent: runs are contiguous, an inclusive maximum up to its last lane
            ey = use ? yf : 0;
            const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, ey, o);
                if (lane - o >= start) ey = max(ey, v);
            }
            const unsigned later = lane < 31 ? heads & (0xfffffffeu << lane) : 0u;
            ey = __shfl_sync(0xffffffffu, ey, (later ? __ffs(later) - 1 : cnt) - 1);
            // y w 2^(61 - e), e = ey - 1022; |w| < 2.  Sums over thousands of samples show a bias, so
            // both products are rounded to nearest, and what is shifted below rounds ties to even.  All of
            // its 62 bits enter the seven digits (1e7 uniform samples on 127 x 128 cells, cube against long
            // double: 5.9e-16; six digits, 2^-53 of twice the run's largest |y|: 16e-16; FP64: 6.7e-16).
            const long long yq = use ? fx_from_double(y, ey) >> 1 : 0;
            // halves of row 4 a + slot from row 4 a on: an odd a flips the third bit of the word (fa_word)
            __half *arow = reinterpret_cast<__half *>(W.a) + (lane & 1);
            int off[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int slot = (j - 1 + b) & 3;
                off[b] = 2 * (slot * kFaRow + fa_word(slot, lane >> 1));
            }
#pragma unroll 1
            for (int a = 0; a < 4; ++a) {
                const long long ya = fx_mul_rn(yq, lwt[0]);
                lwt[0] = lwt[1];
                lwt[1] = lwt[2];
                lwt[2] = lwt[3];
#pragma unroll
                for (int b = 0; b < 4; b += 2) {
                    uint32_t d[kFaDig];
                    fx_digits(fx_mul_rn(ya, lwp[b]), fx_mul_rn(ya, lwp[b + 1]), d);
                    __half *o0 = arow + (off[b] ^ ((a & 1) << 4)), *o1 = arow + (off[b + 1] ^ ((a & 1) << 4));
#pragma unroll
                    for (int u = 0; u < kFaDig; ++u) {
                        const __half2 h = *reinterpret_cast<const __half2 *>(&d[u]);
                        o0[u * (16 * 2 * kFaRow)] = __low2half(h);
                        o1[u * (16 * 2 * kFaRow)] = __high2half(h);
                    }
                }
                arow += 4 * 2 * kFaRow;
            }
        }
        if (t0 + 32 < wlast) {
            s_next = A.perm[min(t0 + 32 + lane, wlast - 1)];
            r_next = A.rec[s_next];
            ps_next = A.psi[s_next];
            y_next = A.y[s_next];
        }
        __half *erow = reinterpret_cast<__half *>(W.e) + (lane & 1);
        long long xc = zc, xs = -zs, pc = kFxOne, px = 0;
        // ---- 2: order 0 (E = 1: the first digit 256 alone, FP16 0x5c00, in column 0), then blocks of
        // four orders
        unsigned cell = cur;
        int e = ecur;
#pragma unroll 1
        for (int b = -1; b < nblk; ++b) {
            if (b >= 0) {
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    uint32_t d[kFxDig];
                    fx_digits(xc, xs, d);
#pragma unroll
                    for (int u = 0; u < kFxDig; ++u) {
                        const __half2 h = *reinterpret_cast<const __half2 *>(&d[u]);
                        __half *o = erow + 2 * ((u * 8 + 2 * k) * kFaRow + fa_word(2 * k, lane >> 1));   // 2 k + 1: the same swizzle
                        o[0] = __low2half(h);
                        o[2 * kFaRow] = __high2half(h);
                    }
                    const long long nc = fx_cheb(zc, xc, pc), ns = fx_cheb(zc, xs, px);
                    pc = xc;
                    px = xs;
                    xc = nc;
                    xs = ns;
                }
            }
            __syncwarp();
            cell = cur;
            e = ecur;
            long long *v = sums + (b < 0 ? 0 : 32 * (2 + 4 * b));
            const int nv = b < 0 ? 2 : 4;
            // runs of equal cells, [r0, r1)
#pragma unroll 1
            for (int r0 = 0, r1; r0 < cnt; r0 = r1) {
                const unsigned rcell = __shfl_sync(0xffffffffu, mycell, r0);
                const int re = __shfl_sync(0xffffffffu, ey, r0);
                const unsigned later = r0 < 31 ? heads & (0xfffffffeu << r0) : 0u;
                r1 = later ? __ffs(later) - 1 : cnt;
                if (re == 0) continue;              // nothing to add
                if (rcell != cell) {
                    if (cell != 0xffffffffu) {
                        const int jo = (int)(cell & 0xffffu), jn = (int)(rcell & 0xffffu);
                        const bool near = (rcell >> 16) == (cell >> 16) && jn > jo && jn < jo + 4;
                        flush(b, cell, e, jo - 1, near ? jn - 1 : jo + 3);
                    }
                    cell = rcell;
                }
                // sums and contributions to one exponent; the products' unit is 2^(re - 1022 + 1)
                const int en = re - 1021;
                int shift = 3;
                if (en > e) {
                    if (e != kFaEmpty) {
                        const int d = en - e;
                        for (int q = 0; q < nv; ++q) v[32 * q] = d > 61 ? 0 : fx_shift_even(v[32 * q], d);
                    }
                    e = en;
                } else {
                    shift = min(3 + e - en, 62);
                }
                float acc[4][kFaDig];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int u = 0; u < kFaDig; ++u) acc[q][u] = 0.f;
                // the run's samples within each half of the batch
#pragma unroll 1
                for (int t = r0 >> 4; t <= (r1 - 1) >> 4; ++t) {
                    const int p0 = 16 * t + 2 * q4, p1 = p0 + 8;
                    const uint32_t m0 = (p0 >= r0 && p0 < r1 ? 0xffffu : 0u) | (p0 + 1 >= r0 && p0 + 1 < r1 ? 0xffff0000u : 0u);
                    const uint32_t m1 = (p1 >= r0 && p1 < r1 ? 0xffffu : 0u) | (p1 + 1 >= r0 && p1 + 1 < r1 ? 0xffff0000u : 0u);
                    const int w0 = fa_word(gr, 8 * t + q4);     // rows gr and gr + 8: the same swizzle
                    uint32_t ad[kFaDig][4];
#pragma unroll
                    for (int u = 0; u < kFaDig; ++u) {
                        ad[u][0] = W.a[u][gr][w0] & m0;
                        ad[u][1] = W.a[u][gr + 8][w0] & m0;
                        ad[u][2] = W.a[u][gr][w0 ^ 4] & m1;
                        ad[u][3] = W.a[u][gr + 8][w0 ^ 4] & m1;
                    }
                    if (b < 0) {
                        const uint32_t one = gr == 0 ? 0x5c005c00u : 0u;
#pragma unroll
                        for (int u = 0; u < kFaDig; ++u)
                            mma_f16(acc[0][u], acc[1][u], acc[2][u], acc[3][u], ad[u], one, one);
                    } else {
#pragma unroll
                        for (int w = 0; w < kFxDig; ++w) {
                            const uint32_t b0 = W.e[w][gr][w0], b1 = W.e[w][gr][w0 ^ 4];
#pragma unroll
                            for (int u = 0; u < kFaDig; ++u)
                                if (u + w < kFaDig)
                                    mma_f16(acc[0][u + w], acc[1][u + w], acc[2][u + w], acc[3][u + w], ad[u], b0, b1);
                        }
                    }
                }
                // (row gr, re), (row gr, im), (row gr + 8, re), (row gr + 8, im); order 0: re only
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const long long c = fx_shift_even(fx_combine(acc[q]), shift);
                    if (b >= 0) v[32 * q] += c;
                    else if (!(q & 1)) v[16 * q] += c;
                }
            }
            __syncwarp();
        }
        cur = cell;
        ecur = e;
    }
    if (cur != 0xffffffffu)
        for (int b = -1; b < nblk; ++b) {
            int e = ecur;
            flush(b, cur, e, (int)(cur & 0xffffu) - 1, (int)(cur & 0xffffu) + 3);
        }
}

SL_CHECK_READER(chk_interp_adj_fx)

// A block of four orders costs 27 mma a run of cells, whatever the run's length, so
// k_interp_adjoint(_df) stays better where the samples leave few per occupied cell.  The sort's count of
// occupied cells tells on the device which kernel runs; the other returns at once (4 us).  Time of the whole
// call over the tiled kernel's, uniform samples, by grid and samples per occupied cell:
//   127 x 128      K = 4: below 0.9 everywhere; K = 8: 1.08 at 4.5, 0.83 at 8.4; K = 16: 1.57, 1.17, 1.16, 0.89 at 4.5, 8.4, 12,
//                  16; K = 32: 1.31, 0.97 at 24, 32 (128 tiles leave most of the chip idle in the tiled kernel)
//   100 x 128      K <= 16: 0.43-0.97 everywhere
//   150 x 200      K = 4: below 1 to 12, 1.2 at 24
//   180 x 200 and 199 x 200 (one wave of tiles)   K = 4: 1.14, 1.1, 1.2, 1.15 / 0.82, 0.7 / 0.8 at 4.5, 12, 16, 24, 32; K = 16: 1.8,
//                  1.35, 1.2, 1.17 / 0.78, 0.67; K = 1: 1.06, 1.25 at 32
//   300 x 600      K = 4, 8, 16: 1.4 and 0.8 at 8.4 and 12; K = 5, 24: 1.18 and 0.94 at 12 and 16; K = 1: 1.06 and 0.90 at 24, 32
//   512 x 1024     K = 4-32: 0.91-1.1 and 0.52-0.8 at 8.4 and 12; K = 1: 1.04 and 0.90 at 12 and 16
//   724 x 1500     K = 4-32: 1.14-1.32, 0.87-1.01 and 0.73-0.82 at 3, 5, 7; K = 2: 0.95 at 7; K = 1: 0.99 at 12
//   1024 x 2048 to 2048 x 4096   K = 4-32: 0.84-1.16 and 0.67-0.90 at 3 and 5; K = 2: 0.77-0.85 at 7; K = 1: 0.73-0.86 at 12
//   the same, 4 to 10 samples in each of 3% or 30% of the cells: K = 2 to 32 0.40-0.91
//   DF64           180 x 200 and 199 x 200: 1.2-2.2 and 1.0-1.4 at 24 and 32; 300 x 600: 0.87-1.04 at 24 (K = 2: 1.17 at 32);
//                  512 x 1024: 0.65-0.83 at 24 (K = 2: 1.01 at 32); 724 x 1500 and more: K = 4-16 1.06-1.33 and 0.61-0.90
//                  at 7 and 12; K = 32 0.83-0.95 at 16
// Small calls: the tiled kernel clears and writes whole tiles, so with 1000 to 16,000 uniform samples this
// one takes 0.4-0.85 of its time on 300 x 600 cells and more; on 250 x 256 it is even at 4000 (1.1-1.2 at 16,000),
// at K = 32 at 2000; on 127 x 128 0.7-1.0.  A scan of 16,000 samples, 13 to 46 per occupied cell, takes 0.3-0.9, of 40,000
// 0.2-0.9: below 131,072 samples uniform ones reach 12 per occupied cell on the smallest grids only.
// The p = 2 and 6 stencils (4 and 36 nodes) do not fill rows of 16, and above 32 orders the sums no
// longer leave two blocks a multiprocessor.
AdjRoute interp_adj_route(const sl_plan *p, int64_t n, float *min_mean) {
    const bool df = p->precision == SL_DF64;
    const int K = p->K;
    const int64_t cells = (int64_t)(p->R + 1) * p->nphi;
    const bool large = cells >= 120000, huge = cells >= 1000000;
    *min_mean = 0.f;
    if (p->p != 4 || K > 32) return AdjRoute::tiled;
    if (n <= (df || K > 16 ? 2048 : 4096) || (large && n <= (df ? 8192 : 16384))) return AdjRoute::fx;
    if (K <= 4 && cells <= 32768 && (cells <= 20000 || n < 12 * cells)) return AdjRoute::fx;
    if (!df && K <= 16 && (cells <= 14000 || (cells <= 20000 && n <= 16384))) return AdjRoute::fx;
    if (n <= 16384) *min_mean = 4.f;
    else if (n <= 131072) *min_mean = 12.f;
    else if (huge && K > 2) *min_mean = !df ? 5.f : K <= 16 ? 12.f : 16.f;
    else if (huge && K == 2 && !df) *min_mean = 7.f;
    else if (df) *min_mean = large && K > 2 ? 24.f : 40.f;
    else if (large) *min_mean = K <= 1 ? (cells < 400000 ? 30.f : 14.f) : cells < 400000 && (K == 5 || K > 16) ? 16.f : 12.f;
    else if (cells > 20000) *min_mean = K <= 1 ? 40.f : 30.f;
    else *min_mean = K <= 12 ? 7.f : K <= 16 ? 14.f : 32.f;
    return (double)n >= *min_mean * (double)cells ? AdjRoute::fx : AdjRoute::by_occupancy;
}

sl_status launch_interp_adj_fx(sl_plan *p, const SortBufs &b, const double *psi, const double *tod, int64_t n, const unsigned *occ,
                               float min_mean, double2 *fbar) {
    FaArgs a;
    a.g = p->geom;
    a.psi = psi;
    a.y = tod;
    a.rec = (const StencilRec64 *)b.rec;
    a.perm = b.perm;
    a.occ = occ;
    a.min_mean = min_mean;
    a.n = n;
    a.fbar = fbar;
    const size_t sm = 256 * sizeof(longlong2) + kFaWarps * fa_warp_bytes((p->K + 3) / 4);
    cudaError_t e = allow_dyn_smem(k_interp_adj_fx, sm);
    if (e != cudaSuccess) return cuda_check(e, "k_interp_adj_fx smem attribute");
    int nsm = 152, per_sm = 1;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_interp_adj_fx, 32 * kFaWarps, sm);
    const int64_t full = (int64_t)nsm * std::max(per_sm, 1) * kFaWarps;     // warps of one wave
    const int64_t waves = std::max<int64_t>(1, (n + full * kFaChunk - 1) / (full * kFaChunk));
    const int64_t per = (n + full * waves - 1) / (full * waves);            // whole waves
    a.chunk = (int)(per <= 32 ? std::max<int64_t>(per, 1) : (per + 31) / 32 * 32);
    const int64_t nwarps = (n + a.chunk - 1) / a.chunk;
    const int slot = timing_begin(p, "interp_adj_fx");
    k_interp_adj_fx<<<(unsigned)((nwarps + kFaWarps - 1) / kFaWarps), 32 * kFaWarps, sm, p->stream>>>(a);
    timing_end(p, slot);
    return cuda_check(cudaGetLastError(), "k_interp_adj_fx launch");
}

}  // namespace sl
