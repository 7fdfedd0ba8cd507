// k_lcontract_fx.cu -- the spin "Legendre" step (Sect. 2.1, Eqs. c_m and S; the sums and
// reflections of k_lcontract.cu) of FP64 plans, in fixed point and on the tensor cores:
//
//   sums of one (m, k, sign of k):   S[ring][c] = sum_l y_l(ring) V_l[c],  c = 0..3
//
// with y the rescaled Wigner values of the recurrence y_{l+1} = (a'_l x - b'_l) y_l - y_{l-1}
// and V the re / im parts of the two sky x beam columns.  In FP64 a step is six operations
// (two for the recurrence, four for the sums) on a pipe that runs at 1/64 of the FP32 rate:
// that form kept it 99% busy for 68.7 ms at lmax 1024, kmax 16, 1024 rings.  Here
//
//   - the sums run on the tensor cores as exact digit products (fxdigits.cuh): the seven
//     9-bit digits of y (16 rings x 8 l per mma.sync m16n8k8) times six digits of V, two
//     digits of the four columns per MMA: 15 MMAs for the pairs of order <= 6 (the odd slots
//     of the last ones give some of order 7, which are dropped).  Four columns fill the N = 8
//     of mma.sync with two digits each; a tcgen05 tile would spend its 128 rows of A reads on
//     the same eight columns, and 0.15 clocks a step are not what binds;
//   - the recurrence runs on the integer pipe in 64-bit fixed point (LfRec): |d| <= 1 and
//     y = d / c with decreasing c bound |y| by 2^U; Y = y 2^(60 - U).  While its rings are
//     still growing out of the evanescent zone (they start at 2^-64, where fixed point would
//     lose the leading digits), and near l = max(m, k), where a' + |b'| >= 4, a warp's
//     recurrences run in FP64, two operations a step.  The two forms share the work about
//     equally, which suits two pipes.
//
// Measured at that size: 28.1 ms, FP64 pipe 66%, integer ALU 58% busy (about 80 instructions
// a step, 4 warps per scheduler).  Against long double the errors are those of the FP64 form
// (set by the rounding of a' and b'), or smaller: 5.7e-16 against 1.5e-15 over the far
// sidelobe beam's G.  Tried: an exponent per ring instead of FP64 for the growing part (40 ms,
// 14 more instructions a step), five warps of 96 registers per scheduler (30.2 ms, spills),
// the two forms unrolled over 8 l (35 ms, instruction cache).
//
// Each warp is independent: units of 32 ring pairs (both signs of k of 16 pairs side by side,
// two such groups one after the other) from their earliest start l, in batches of 64 l.  Per
// batch a lane forms V and the coefficients of two l (FP64) and the warp scales V by its
// largest value; the digit sums are read out after each batch (64 l keep |acc| < 2^24) and
// added in FP64.
//
// A batch with a non-finite V, or one above 2^960, sends the whole unit to the plain FP64 loop (the
// sums then overflow or turn NaN where that form does).  One whose largest V is below 2^-959 (the
// tail of a Gaussian beam: exp(-l^2 / 2 sigma^2) from l = 36 sigma on) is summed times 2^600, unless sums
// above 2^400 stand there already: in the plain loop, lmax 2048, kmax 32 with such a beam took
// 1968 ms, 981 in the FP64 form, 401 so.
#include <algorithm>

#include "lcontract.cuh"
#include "lfrec.cuh"

namespace sl {

constexpr int kLfWarps = 4;        // warps per CTA, four CTAs per SM (128 registers a thread)
constexpr int kLfBatch = 64;       // l per batch

struct LfWarp {                    // one warp's shared memory
    uint32_t yd[7][4][32];         // digits of y at 8 l: [digit][pair of l][ring], swizzled (lf_slot)
    uint32_t vf[kLfBatch / 8][3][32];   // B fragments of V: [8 l][digit pair][lane]
    int4 ci[kLfBatch];             // a' 2^58 as (Ah, Al), -b' 2^58 (LfRec)
    double2 cd[kLfBatch];          // a', -b'
    // per group and lane: the recurrence's values at l - 1 and l, as doubles or in fixed point;
    // before the start l: the start state
    longlong2 state[2][32];
    int ls[2][32];                 // start l << 1 | has grown to 2^(U - 7)
    double2 sum[2][2][32];         // FP64 sums of this lane's ring and column pair, per group and row tile
};

// Ring r's slot in the row of l pair p: the rows of a fragment's four pairs in distinct banks.
__device__ __forceinline__ int lf_slot(int p, int r) { return r ^ ((p & 3) << 3); }

// V of one l: (c ap, (-1)^l c am) as re and im, ap = sum s conj(b), am = sum conj(s) conj(b).
// It serves both signs of k: (-1)^l d_{m,-k}(theta) follows the recurrence of +k at
// x = -cos theta, and with y' = (-1)^l y the -k sums of c am y and (-1)^l c ap y are those of
// V's second and first column with y'.
__device__ __forceinline__ void lf_columns(const LcArgs &a, int64_t moff, int m, int k, int l, double c, double v[4]) {
    double p = 0.0, q = 0.0, r = 0.0, t = 0.0;
    for (int X = 0; X < a.ncomp; ++X) {
        double2 s = a.sky[X * a.nalm + moff + l];
        if (m == 0) s.y = 0.0;
        double2 b = a.beam[((int64_t)X * (a.K + 1) + k) * (a.L + 1) + l];
        if (k == 0) b.y = 0.0;
        p = fma(s.x, b.x, p);
        q = fma(s.y, b.y, q);
        r = fma(s.y, b.x, r);
        t = fma(s.x, b.y, t);
    }
    const double sc = (l & 1) ? -c : c;
    v[0] = c * (p + q);
    v[1] = c * (r - t);
    v[2] = sc * (p - q);
    v[3] = -sc * (r + t);
}

__device__ __forceinline__ void lf_store(LfWarp &W, int pr, int lane, long long v0, long long v1) {
    uint32_t d[7];
    lf_digits(v0, v1, d);
    uint32_t *o = &W.yd[0][pr][lf_slot(pr, lane)];
#pragma unroll
    for (int j = 0; j < 7; ++j) o[128 * j] = d[j];
}

// The plain FP64 loop of one ring, out of line (rare).
__device__ __noinline__ void lf_plain(const LcArgs &a, int m, int k, int pair, int neg) {
    if (pair >= a.npairs) return;
    const int64_t moff = (int64_t)m * (2 * a.L + 1 - m) / 2, si = start_index(a, k, m, neg, pair);
    const RTab64 *tab = a.tab64 + (int64_t)k * a.nalm + moff;
    double yo = a.st64[si].x, y = a.st64[si].y;
    const double x = a.xr[pair];
    double2 acc1 = {0, 0}, acc2 = {0, 0};
    for (int l = a.ls[si]; l <= a.L; ++l) {
        const RTab64 t = tab[l];
        double v[4];
        lf_columns(a, moff, m, k, l, t.c, v);
        const double ys = (neg && (l & 1)) ? -y : y;
        acc1.x = fma(v[0], ys, acc1.x);
        acc1.y = fma(v[1], ys, acc1.y);
        acc2.x = fma(v[2], ys, acc2.x);
        acc2.y = fma(v[3], ys, acc2.y);
        const double yn = fma(fma(t.a, x, neg ? t.b : -t.b), y, -yo);
        yo = y;
        y = yn;
    }
    write_one(a, m, k, pair, neg, neg, acc1);
    write_one(a, m, k, pair, neg, 1 - neg, acc2);
}

// One batch of 64 l from c0 for one group: 16 ring pairs, +k in lanes 0-15, -k in lanes 16-31
// (x: +-cos theta).  fixed: the group's recurrences run in fixed point.
__device__ __forceinline__ void lf_batch(const LcArgs &a, LfWarp &W, int grp, bool &fixed, double x, int U,
                                         int c0, uint64_t steep, int escale) {
    const int lane = threadIdx.x & 31, gr = lane >> 2, q4 = lane & 3;
    const int ls = W.ls[grp][lane] >> 1;
    bool grown = W.ls[grp][lane] & 1;
    double y = 0.0, yo = 0.0;
    LfRec r;
    r.Y = r.Yo = 0;
    lf_set_x(r, x);
    const longlong2 st = W.state[grp][lane];
    const double so = __longlong_as_double(st.x), sv = __longlong_as_double(st.y);
    if (fixed) {
        r.Yo = st.x;
        r.Y = st.y;
    } else if (ls < c0) {
        yo = so;
        y = sv;
    }
    const double big = __longlong_as_double((long long)(1023 + U - 7) << 52);

    float acc[2][7][4];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int s = 0; s < 7; ++s)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[t][s][e] = 0.f;
#pragma unroll 1
    for (int ks = 0; ks < kLfBatch / 8 && c0 + 8 * ks <= a.L; ++ks) {
        const int lk = c0 + 8 * ks;
        // once every ring has grown to 2^(U - 7), where a unit of the fixed point is 2^-52 of it; not
        // before a' + |b'| < 4 from here on
        grown |= ls < lk && fmax(fabs(y), fabs(yo)) >= big;
        if (!fixed && !(steep >> (8 * ks)) && __all_sync(0xffffffffu, grown || ls > a.L)) {
            fixed = true;
            r.Y = lf_from_double(y, U);
            r.Yo = lf_from_double(yo, U);
        }
        // two l per round, rolled: unrolled, the two forms do not fit the instruction cache
        if (fixed) {
            const int4 *cf = W.ci + 8 * ks;
#pragma unroll 1
            for (int pr = 0; pr < 4; ++pr) {
                const long long v0 = r.Y;
                r.step(cf[2 * pr]);
                const long long v1 = r.Y;
                r.step(cf[2 * pr + 1]);
                lf_store(W, pr, lane, v0, v1);
            }
        } else {
#pragma unroll 1
            for (int pr = 0; pr < 4; ++pr) {
                long long v[2];
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const int l = lk + 2 * pr + o;
                    const double2 ab = W.cd[8 * ks + 2 * pr + o];
                    if (l == ls) {
                        yo = so;
                        y = sv;
                    }
                    v[o] = fx_from_double(y, U + 1024);
                    const double yn = fma(fma(ab.x, x, ab.y), y, -yo);
                    yo = y;
                    y = yn;
                }
                lf_store(W, pr, lane, v[0], v[1]);
            }
        }
        __syncwarp();
        const uint32_t b0 = W.vf[ks][0][lane], b1 = W.vf[ks][1][lane], b2 = W.vf[ks][2][lane];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                const uint32_t a0 = W.yd[i][q4][lf_slot(q4, 16 * t + gr)], a1 = W.yd[i][q4][lf_slot(q4, 16 * t + gr + 8)];
                mma_f16_k8(acc[t][i], a0, a1, b0);
                if (i + 2 < 7) mma_f16_k8(acc[t][i + 2], a0, a1, b1);
                if (i + 4 < 7) mma_f16_k8(acc[t][i + 4], a0, a1, b2);
            }
        __syncwarp();
    }
    W.ls[grp][lane] = (ls << 1) | (int)grown;
    if (fixed) W.state[grp][lane] = make_longlong2(r.Yo, r.Y);
    else if (ls < c0 + kLfBatch) W.state[grp][lane] = make_longlong2(__double_as_longlong(yo), __double_as_longlong(y));
    // Read out: columns 0-3 (lanes q4 < 2) hold the even digits of V, columns 4-7 the odd ones,
    // 2^-9 lower.  In units of 2^-34 (orders 0-2) and 2^-70 (orders 3-6; the odd columns' order 7
    // is dropped).  Lanes q4 < 2 go on with row gr, the others with row gr + 8; both with the
    // column pair q4 & 1.
    const bool odd = q4 >= 2;
    const int h0 = odd ? 1 << 9 : 1 << 18, h1 = odd ? 1 : 1 << 9, h2 = odd ? 0 : 1;
    const int w2 = odd ? 1 << 27 : 0, w3 = odd ? 1 << 18 : 1 << 27, w4 = odd ? 1 << 9 : 1 << 18, w5 = odd ? 1 : 1 << 9,
              w6 = odd ? 0 : 1;
    const double sc = __longlong_as_double((long long)(escale + U + 1 - 34) << 52);     // 2^(U + e - 34), e = escale - 1022
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        long long H[4], Lw[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            int w[7];
#pragma unroll
            for (int s = 0; s < 7; ++s) w[s] = __float2int_rn(acc[t][s][e]);
            H[e] = (long long)w[0] * h0 + (long long)w[1] * h1 + (long long)w[2] * h2;
            Lw[e] = (long long)w[2] * w2 + (long long)w[3] * w3 + (long long)w[4] * w4 + (long long)w[5] * w5 + (long long)w[6] * w6;
        }
        double2 s = W.sum[grp][t][lane];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const long long h = (odd ? H[2 + e] : H[e]) + __shfl_xor_sync(0xffffffffu, odd ? H[e] : H[2 + e], 2);
            const long long l = (odd ? Lw[2 + e] : Lw[e]) + __shfl_xor_sync(0xffffffffu, odd ? Lw[e] : Lw[2 + e], 2);
            double &o = e ? s.y : s.x;
            o = fma((double)l, sc * 0x1p-36, o);
            o = fma((double)h, sc, o);
        }
        W.sum[grp][t][lane] = s;
    }
}

// This lane's sums times f, for a batch of tiny V; false, in every lane, if one would overflow.  Out of line
// (rare): 2^600 applied as the sums are read out cost every batch 2% of the kernel.
__device__ __noinline__ bool lf_scale_sums(LfWarp &W, int groups, double f) {
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int grp = 0; grp < groups; ++grp)
        for (int t = 0; t < 2; ++t) {
            double2 &s = W.sum[grp][t][lane];
            ok = ok && fabs(s.x) < 0x1p400 && fabs(s.y) < 0x1p400;
            s = make_double2(s.x * f, s.y * f);
        }
    return __all_sync(0xffffffffu, ok);
}

// One unit: (m, k, 16 groups ring pairs); 2 groups (V staged once for both) or 1.
__device__ __forceinline__ void lf_unit(const LcArgs &a, LfWarp &W, int groups, unsigned u) {
    const int lane = threadIdx.x & 31;
    const unsigned nchunk = (unsigned)(a.npairs + 16 * groups - 1) / (16u * groups);
    const int base = 16 * groups * (int)(u % nchunk);
    u /= nchunk;
    const int k = (int)(u % (unsigned)(a.K + 1)), m = (int)(u / (unsigned)(a.K + 1));
    const int neg = lane >> 4;
    const int64_t moff = (int64_t)m * (2 * a.L + 1 - m) / 2;
    const RTab64 *tab = a.tab64 + (int64_t)k * a.nalm + moff;
    const int gr = lane >> 2, q4 = lane & 3;

    double x0 = 0.0, x1 = 0.0;
    int lstart = a.L + 1, lfirst1 = a.L + 1;
    for (int grp = 0; grp < groups; ++grp) {
        const int pair = base + 16 * grp + (lane & 15);
        int ls = a.L + 1;
        double x = 0.0;
        double2 st = make_double2(0.0, 0.0);
        if (pair < a.npairs) {
            const int64_t si = start_index(a, k, m, neg, pair);
            ls = a.ls[si];
            st = a.st64[si];
            x = a.xr[pair];
            if (neg) {                  // -k: (-1)^l times the state, at -x
                x = -x;
                if (ls & 1) st.y = -st.y;
                else st.x = -st.x;
            }
        }
        W.state[grp][lane] = make_longlong2(__double_as_longlong(st.x), __double_as_longlong(st.y));
        W.ls[grp][lane] = ls << 1;
        W.sum[grp][0][lane] = W.sum[grp][1][lane] = make_double2(0.0, 0.0);
        const int lf = __reduce_min_sync(0xffffffffu, ls);
        lstart = min(lstart, lf);
        if (grp) {
            x1 = x;
            lfirst1 = lf;
        } else {
            x0 = x;
        }
    }
    double cmin = tab[a.L].c;
    if (a.L > max(m, k)) cmin = fmin(cmin, tab[a.L - 1].c);
    const int U = lf_bound(cmin);
    const int lfirst0 = __reduce_min_sync(0xffffffffu, W.ls[0][lane] >> 1);
    bool fixed0 = false, fixed1 = false;

    for (int c0 = lstart; c0 <= a.L; c0 += kLfBatch) {
        // ---- V and the coefficients of the batch, two l per lane
        double v[2][4];
        uint32_t mx = 0;
        uint64_t steep = 0;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 32 * h + lane, l = c0 + i;
            RTab64 t = {0.0, 0.0, 0.0, 0.0};
            v[h][0] = v[h][1] = v[h][2] = v[h][3] = 0.0;
            if (l <= a.L) {
                t = tab[l];
                lf_columns(a, moff, m, k, l, t.c, v[h]);
            }
            W.cd[i] = make_double2(t.a, -t.b);
            bool big;                   // the batch's FP64 steps cover these (a' + |b'| falls over every second l)
            W.ci[i] = lf_coef(t.a, t.b, big);
            steep |= (uint64_t)__ballot_sync(0xffffffffu, big) << (32 * h);
#pragma unroll
            for (int c = 0; c < 4; ++c) mx = max(mx, (uint32_t)__double2hiint(v[h][c]) & 0x7fffffffu);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        int escale = (int)(mx >> 20);   // exponent field of the largest |V|
        bool plain = escale > 1983, tiny = false;
        if (escale < 64) {              // all zero (any scale), or too small for one: V and the sums times 2^600
            mx = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    v[h][c] *= 0x1p600;
                    mx = max(mx, (uint32_t)__double2hiint(v[h][c]) & 0x7fffffffu);
                }
            escale = (int)(__reduce_max_sync(0xffffffffu, mx) >> 20);
            tiny = escale > 0;
            escale = max(escale, 64);
            if (tiny) plain = !lf_scale_sums(W, groups, 0x1p600);
        }
        if (plain) {
            for (int grp = 0; grp < groups; ++grp) lf_plain(a, m, k, base + 16 * grp + (lane & 15), neg);
            return;
        }
        // digits, to the B fragment of each 8 l: element (l, column n), n = digit parity * 4 + c, in
        // lane 4 n + (l % 8) / 2, half l % 2
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 32 * h + lane;
            __half *row = reinterpret_cast<__half *>(W.vf[i >> 3][0]) + (i & 7);
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                uint32_t d[kFxDig];
                fx_digits(fx_from_double(v[h][c], escale), fx_from_double(v[h][c + 1], escale), d);
#pragma unroll
                for (int j = 0; j < kFxDig; ++j) {
                    const int ln = 4 * ((j & 1) * 4 + c);
                    const __half2 hd = *reinterpret_cast<const __half2 *>(&d[j]);
                    row[((j >> 1) * 32 + ln) * 2] = __low2half(hd);
                    row[((j >> 1) * 32 + ln + 4) * 2] = __high2half(hd);
                }
            }
        }
        __syncwarp();
        // ---- the recurrences and sums of each group that has begun
#pragma unroll 1
        for (int grp = 0; grp < groups; ++grp) {
            if ((grp ? lfirst1 : lfirst0) >= c0 + kLfBatch) continue;
            bool fixed = grp ? fixed1 : fixed0;
            lf_batch(a, W, grp, fixed, grp ? x1 : x0, U, c0, steep, escale);
            if (grp) fixed1 = fixed;
            else fixed0 = fixed;
        }
        if (tiny) lf_scale_sums(W, groups, 0x1p-600);
    }
    __syncwarp();
    for (int grp = 0; grp < groups; ++grp)
#pragma unroll
        for (int t = 0; t < 2; ++t) {   // row tile t: sign t; columns: the -k sums are exchanged
            const int r = base + 16 * grp + gr + (q4 >= 2 ? 8 : 0);
            if (r < a.npairs) write_one(a, m, k, r, t, (q4 & 1) ^ t, W.sum[grp][t][lane]);
        }
}

// Units in order of m (the longest l ranges first), claimed from *counter by the resident
// warps (counter null: one unit per warp).
__global__ void __launch_bounds__(32 * kLfWarps, 4) k_lcontract_fx(const __grid_constant__ LcArgs a, int groups, unsigned nunits,
                                                                   unsigned *counter) {
    extern __shared__ __align__(16) unsigned char lf_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LfWarp &W = reinterpret_cast<LfWarp *>(lf_smem)[warp];
    unsigned u = blockIdx.x * kLfWarps + warp;
    if (counter) {
        if (lane == 0) u = atomicAdd(counter, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
    }
    while (u < nunits) {
        unsigned next = 0xffffffffu;    // claimed before this unit runs: the atomic's round trip overlaps it
        if (counter && lane == 0) next = atomicAdd(counter, 1u);
        lf_unit(a, W, groups, u);
        __syncwarp();
        u = __shfl_sync(0xffffffffu, next, 0);
    }
}

sl_status launch_lcontract_fx(sl_plan *p, const LcArgs &a) {
    const size_t sm = kLfWarps * sizeof(LfWarp);
    cudaError_t e = allow_dyn_smem(k_lcontract_fx, sm);
    if (e != cudaSuccess) return cuda_check(e, "k_lcontract_fx smem attribute");
    // 32 ring pairs per warp where that leaves several warps for every slot
    int nsm = 152;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
    const int64_t mk = (int64_t)(p->L + 1) * (p->K + 1);
    const int groups = mk * ((p->npairs + 31) / 32) >= (int64_t)nsm * 4 * kLfWarps * 4 ? 2 : 1;
    const int64_t nunits = mk * ((p->npairs + 16 * groups - 1) / (16 * groups)), slots = (int64_t)nsm * 4 * kLfWarps;
    if (nunits > 0x7fffffff) return set_error(SL_ERR_UNSUPPORTED, "grid too large");
    unsigned *counter = nullptr;
    if (nunits > slots) {
        counter = p->d_lc_counter;
        if ((e = cudaMemsetAsync(counter, 0, sizeof(unsigned), p->stream)) != cudaSuccess) return cuda_check(e, "unit counter");
    }
    const unsigned nblk = (unsigned)((std::min(nunits, slots) + kLfWarps - 1) / kLfWarps);
    const int slot = timing_begin(p, "lcontract_fx");
    k_lcontract_fx<<<nblk, 32 * kLfWarps, sm, p->stream>>>(a, groups, (unsigned)nunits, counter);
    timing_end(p, slot);
    return cuda_check(cudaGetLastError(), "k_lcontract_fx launch");
}

}  // namespace sl
