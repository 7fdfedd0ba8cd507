// k_adjoint_fx.cu -- transpose of the spin "Legendre" step (the sums of k_adjoint.cu) in
// fixed point and on the tensor cores, for every plan (the adjoint of FP32 plans runs with
// FP64 tables and accuracy):
//
//   Abar_{+m}(l) = c_l P_l[0],   Abar_{-m}(l) = (-1)^l c_l P_l[1],
//   P_l[c] = sum over rings and signs of k of y'_l(ring) g_c(ring)
//
// with y' the recurrence values of k_lcontract_fx.cu ((-1)^l times those of -k) and g the
// ring's two Ghat values: for +k Ghat(N, +m) and (-1)^k Ghat(S, -m), for -k (-1)^m Ghat(S, +m)
// and (-1)^{m+k} Ghat(N, -m).
//
// The FP64 form was bound by the FP64 pipe (88.3 ms at lmax 1024, kmax 16, 1024 rings: two
// operations of recurrence and four of dot products a step, run in lock step from the CTA's
// earliest start).  Here the recurrence is that of k_lcontract_fx.cu (fixed point, FP64 while
// the rings grow), and the dot products are digit products on mma.sync m16n8k16: 16 l x 16
// rings of the seven digits of y against six digits of g, whose fragments a warp keeps in
// shared memory for all l.  The digit sums are read out after every 16 l (64 rings: at most
// 64 terms keep |acc| < 2^24) and added to Abar atomically, as the CTAs of the FP64 form did.
// 26.1 ms at that size (double-float form of DF64 plans, 78 instructions a step, before: 28.5
// ms); 22.5 us against 71.7 at lmax 64, kmax 4.  g is scaled by its largest value over the unit's rings; a
// non-finite one, or one outside 2^-959 .. 2^960, sends the unit to a plain FP64 loop.
#include <algorithm>

#include "lcontract.cuh"
#include "lfrec.cuh"

namespace sl {

constexpr int kAfWarps = 4;        // warps per CTA, four CTAs per SM (128 registers a thread)
constexpr int kAfBatch = 64;       // l whose coefficients are staged together

struct AfArgs {
    int L, K, R, npairs;
    int64_t nalm;
    const double *xr;
    const int *ls;
    const double2 *st64;
    const RTab64 *tab;
    const double2 *Ghat;           // [K+1][R][2L+1]
    double2 *Abar;                 // [K+1][2L+1][L+1], zeroed
};

struct AfWarp {                    // one warp's shared memory
    uint32_t yd[7][16][16];        // digits of y at 16 l: [digit][l][pair of rings], swizzled (af_word)
    uint2 gf[2][2][3][32];         // B fragments of g: [group][16 rings][digit pair][lane]
    int4 ci[kAfBatch];             // coefficients for LfRec
    double2 cd[kAfBatch];          // a', -b'
    double c[kAfBatch];            // c_l
    longlong2 state[2][32];        // as LfWarp
    int ls[2][32];
};

// Word w of row l: the rows of an A fragment's column pairs in distinct banks.
__device__ __forceinline__ int af_word(int l, int w) { return w ^ (((l >> 1) & 3) << 2); }

// The two Ghat values of one ring and sign of k.
__device__ __forceinline__ void af_partners(const AfArgs &a, int m, int k, int pair, int neg, double2 &g0, double2 &g1) {
    g0 = g1 = make_double2(0.0, 0.0);
    if (pair >= a.npairs) return;
    const int rn = pair, rs = a.R - 1 - pair;
    const int64_t row = 2 * (int64_t)a.L + 1;
    const double2 *Gk = a.Ghat + (int64_t)k * a.R * row;
    if (!neg) {
        g0 = Gk[rn * row + a.L + m];
        if (m > 0 && rs != rn) g1 = Gk[rs * row + a.L - m];
        if (k & 1) g1 = make_double2(-g1.x, -g1.y);
    } else {
        if (rs != rn) g0 = Gk[rs * row + a.L + m];
        if (m & 1) g0 = make_double2(-g0.x, -g0.y);
        if (m > 0) g1 = Gk[rn * row + a.L - m];
        if ((m ^ k) & 1) g1 = make_double2(-g1.x, -g1.y);
    }
}

// Adds c_l P_l[which] to Abar.
__device__ __forceinline__ void af_add(const AfArgs &a, int m, int k, int l, int which, double re, double im) {
    if (which && m == 0) return;
    double2 *o = a.Abar + ((int64_t)k * (2 * a.L + 1) + (which ? a.L - m : a.L + m)) * (a.L + 1) + l;
    atomicAdd(&o->x, re);
    atomicAdd(&o->y, im);
}

// The plain FP64 loop of one ring and sign, out of line (rare).
__device__ __noinline__ void af_plain(const AfArgs &a, int m, int k, int pair, int neg) {
    if (pair >= a.npairs) return;
    const int64_t si = (((int64_t)k * (a.L + 1) + m) * 2 + neg) * a.npairs + pair;
    const RTab64 *tab = a.tab + (int64_t)k * a.nalm + (int64_t)m * (2 * a.L + 1 - m) / 2;
    double yo = a.st64[si].x, y = a.st64[si].y;
    const double x = a.xr[pair];
    double2 g0, g1;
    af_partners(a, m, k, pair, neg, g0, g1);
    for (int l = a.ls[si]; l <= a.L; ++l) {
        const RTab64 t = tab[l];
        const double s = (l & 1) ? -t.c : t.c, v0 = (neg ? s : t.c) * y, v1 = (neg ? t.c : s) * y;
        af_add(a, m, k, l, 0, v0 * g0.x, v0 * g0.y);
        af_add(a, m, k, l, 1, v1 * g1.x, v1 * g1.y);
        const double yn = fma(fma(t.a, x, neg ? t.b : -t.b), y, -yo);
        yo = y;
        y = yn;
    }
}

__device__ __forceinline__ void af_store(AfWarp &W, int pr, int lane, long long v0, long long v1) {
    uint32_t d[7];
    lf_digits(v0, v1, d);
    __half *o = reinterpret_cast<__half *>(&W.yd[0][2 * pr][af_word(2 * pr, lane >> 1)]) + (lane & 1);
#pragma unroll
    for (int j = 0; j < 7; ++j) {      // the rows 2 pr and 2 pr + 1 have the same swizzle
        const __half2 h = *reinterpret_cast<const __half2 *>(&d[j]);
        o[512 * j] = __low2half(h);
        o[512 * j + 32] = __high2half(h);
    }
}

// 16 l from lk of one group's recurrences (16 ring pairs, +k in lanes 0-15, -k in 16-31; x:
// +-cos theta), digits to yd.
__device__ __forceinline__ void af_recur(const AfArgs &a, AfWarp &W, int grp, bool &fixed, double x, int U, int lk, int i0,
                                         bool gentle) {
    const int lane = threadIdx.x & 31;
    const int ls = W.ls[grp][lane] >> 1;
    bool grown = W.ls[grp][lane] & 1;
    const longlong2 st = W.state[grp][lane];
    const double so = __longlong_as_double(st.x), sv = __longlong_as_double(st.y);
    double y = 0.0, yo = 0.0;
    LfRec r;
    r.Y = r.Yo = 0;
    lf_set_x(r, x);
    if (fixed) {
        r.Yo = st.x;
        r.Y = st.y;
    } else if (ls < lk) {
        yo = so;
        y = sv;
    }
    // as k_lcontract_fx: fixed point once every ring has grown to 2^(U - 7) and a' + |b'| < 4
    grown |= ls < lk && fmax(fabs(y), fabs(yo)) >= __longlong_as_double((long long)(1023 + U - 7) << 52);
    if (!fixed && gentle && __all_sync(0xffffffffu, grown || ls > a.L)) {
        fixed = true;
        r.Y = lf_from_double(y, U);
        r.Yo = lf_from_double(yo, U);
    }
    if (fixed) {
        const int4 *cf = W.ci + i0;
#pragma unroll 1
        for (int pr = 0; pr < 8; ++pr) {
            const long long v0 = r.Y;
            r.step(cf[2 * pr]);
            const long long v1 = r.Y;
            r.step(cf[2 * pr + 1]);
            af_store(W, pr, lane, v0, v1);
        }
        W.state[grp][lane] = make_longlong2(r.Yo, r.Y);
    } else {
#pragma unroll 1
        for (int pr = 0; pr < 8; ++pr) {
            long long v[2];
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const double2 ab = W.cd[i0 + 2 * pr + o];
                if (lk + 2 * pr + o == ls) {
                    yo = so;
                    y = sv;
                }
                v[o] = fx_from_double(y, U + 1024);
                const double yn = fma(fma(ab.x, x, ab.y), y, -yo);
                yo = y;
                y = yn;
            }
            af_store(W, pr, lane, v[0], v[1]);
        }
        if (ls < lk + 16) W.state[grp][lane] = make_longlong2(__double_as_longlong(yo), __double_as_longlong(y));
    }
    W.ls[grp][lane] = (ls << 1) | (int)grown;
}

// One unit: (m, k, 16 groups ring pairs); 2 groups or 1.
__device__ __forceinline__ void af_unit(const AfArgs &a, AfWarp &W, int groups, unsigned u) {
    const int lane = threadIdx.x & 31, gr = lane >> 2, q4 = lane & 3, neg = lane >> 4;
    const unsigned nchunk = (unsigned)(a.npairs + 16 * groups - 1) / (16u * groups);
    const int base = 16 * groups * (int)(u % nchunk);
    u /= nchunk;
    const int k = (int)(u % (unsigned)(a.K + 1)), m = (int)(u / (unsigned)(a.K + 1));
    const RTab64 *tab = a.tab + (int64_t)k * a.nalm + (int64_t)m * (2 * a.L + 1 - m) / 2;

    // ---- start states, and g with its scale over the unit
    double x0 = 0.0, x1 = 0.0;
    int lstart = a.L + 1, lfirst0 = a.L + 1, lfirst1 = a.L + 1;
    double2 g[2][2];
    uint32_t mx = 0;
    bool any = false;
#pragma unroll
    for (int grp = 0; grp < 2; ++grp) {
        int ls = a.L + 1;
        double x = 0.0;
        double2 st = make_double2(0.0, 0.0);
        const int pair = base + 16 * grp + (lane & 15);
        g[grp][0] = g[grp][1] = make_double2(0.0, 0.0);
        if (grp < groups && pair < a.npairs) {
            const int64_t si = (((int64_t)k * (a.L + 1) + m) * 2 + neg) * a.npairs + pair;
            ls = a.ls[si];
            st = a.st64[si];
            x = a.xr[pair];
            if (neg) {                  // -k: (-1)^l times the state, at -x
                x = -x;
                if (ls & 1) st.y = -st.y;
                else st.x = -st.x;
            }
            af_partners(a, m, k, pair, neg, g[grp][0], g[grp][1]);
        }
        W.state[grp][lane] = make_longlong2(__double_as_longlong(st.x), __double_as_longlong(st.y));
        W.ls[grp][lane] = ls << 1;
        const int lf = __reduce_min_sync(0xffffffffu, ls);
        lstart = min(lstart, lf);
        if (grp) {
            x1 = x;
            lfirst1 = lf;
        } else {
            x0 = x;
            lfirst0 = lf;
        }
        if (ls <= a.L) {                // rings that never start contribute nothing
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                mx = max(mx, max((uint32_t)__double2hiint(g[grp][c].x) & 0x7fffffffu,
                                 (uint32_t)__double2hiint(g[grp][c].y) & 0x7fffffffu));
                any |= g[grp][c].x != 0.0 || g[grp][c].y != 0.0;
            }
        } else {
            g[grp][0] = g[grp][1] = make_double2(0.0, 0.0);
        }
    }
    if (!__any_sync(0xffffffffu, any)) return;
    mx = __reduce_max_sync(0xffffffffu, mx);
    const int escale = (int)(mx >> 20);
    if (escale < 64 || escale > 1983) {
        for (int grp = 0; grp < groups; ++grp) af_plain(a, m, k, base + 16 * grp + (lane & 15), neg);
        return;
    }
    // digits to the B fragments: element (ring, column n), n = digit parity * 4 + c, in lane
    // 4 n + (ring % 8) / 2, register (ring % 16) / 8, half ring % 2
#pragma unroll
    for (int grp = 0; grp < 2; ++grp) {
        __half *row = reinterpret_cast<__half *>(W.gf[grp][lane >> 4][0]) + ((lane >> 3) & 1) * 2 + (lane & 1) + 4 * ((lane & 7) >> 1);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t d[kFxDig];
            fx_digits(fx_from_double(g[grp][c].x, escale), fx_from_double(g[grp][c].y, escale), d);
#pragma unroll
            for (int j = 0; j < kFxDig; ++j) {
                const int ln = 4 * ((j & 1) * 4 + 2 * c);
                const __half2 hd = *reinterpret_cast<const __half2 *>(&d[j]);
                row[((j >> 1) * 32 + ln) * 4] = __low2half(hd);
                row[((j >> 1) * 32 + ln + 4) * 4] = __high2half(hd);
            }
        }
    }
    double cmin = tab[a.L].c;
    if (a.L > max(m, k)) cmin = fmin(cmin, tab[a.L - 1].c);
    const int U = lf_bound(cmin);
    bool fixed0 = false, fixed1 = false;

    // as in k_lcontract_fx's read-out: column pairs of even and odd digits
    const bool odd = q4 >= 2;
    const int h0 = odd ? 1 << 9 : 1 << 18, h1 = odd ? 1 : 1 << 9, h2 = odd ? 0 : 1;
    const int w2 = odd ? 1 << 27 : 0, w3 = odd ? 1 << 18 : 1 << 27, w4 = odd ? 1 << 9 : 1 << 18, w5 = odd ? 1 : 1 << 9,
              w6 = odd ? 0 : 1;
    const double sc = __longlong_as_double((long long)(escale + U + 1 - 34) << 52);     // 2^(U + e - 34), e = escale - 1022

    for (int c0 = lstart; c0 <= a.L; c0 += kAfBatch) {
        uint64_t steep = 0;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 32 * h + lane, l = c0 + i;
            RTab64 t = {0.0, 0.0, 0.0, 0.0};
            if (l <= a.L) t = tab[l];
            W.cd[i] = make_double2(t.a, -t.b);
            W.c[i] = t.c;
            bool big;
            W.ci[i] = lf_coef(t.a, t.b, big);
            steep |= (uint64_t)__ballot_sync(0xffffffffu, big) << (32 * h);
        }
        __syncwarp();
#pragma unroll 1
        for (int ks = 0; ks < kAfBatch / 16 && c0 + 16 * ks <= a.L; ++ks) {
            const int lk = c0 + 16 * ks;
            float acc[7][4];
#pragma unroll
            for (int s = 0; s < 7; ++s)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[s][e] = 0.f;
#pragma unroll 1
            for (int grp = 0; grp < groups; ++grp) {
                if ((grp ? lfirst1 : lfirst0) >= lk + 16) continue;
                bool fixed = grp ? fixed1 : fixed0;
                af_recur(a, W, grp, fixed, grp ? x1 : x0, U, lk, 16 * ks, !(steep >> (16 * ks)));
                if (grp) fixed1 = fixed;
                else fixed0 = fixed;
                __syncwarp();
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const uint2 b0 = W.gf[grp][t][0][lane], b1 = W.gf[grp][t][1][lane], b2 = W.gf[grp][t][2][lane];
#pragma unroll
                    for (int i = 0; i < 7; ++i) {
                        // rows gr and gr + 8 (the same swizzle), rings 16 t + 2 q4 + {0, 1}, + 8
                        const int wa = af_word(gr, 8 * t + q4), wb = af_word(gr, 8 * t + q4 + 4);
                        const uint32_t A[4] = {W.yd[i][gr][wa], W.yd[i][gr + 8][wa], W.yd[i][gr][wb], W.yd[i][gr + 8][wb]};
                        mma_f16(acc[i][0], acc[i][1], acc[i][2], acc[i][3], A, b0.x, b0.y);
                        if (i + 2 < 7) mma_f16(acc[i + 2][0], acc[i + 2][1], acc[i + 2][2], acc[i + 2][3], A, b1.x, b1.y);
                        if (i + 4 < 7) mma_f16(acc[i + 4][0], acc[i + 4][1], acc[i + 4][2], acc[i + 4][3], A, b2.x, b2.y);
                    }
                }
                __syncwarp();
            }
            // lanes q4 < 2 go on with l = lk + gr, the others with lk + gr + 8; both with P[q4 & 1]
            long long H[4], Lw[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                int w[7];
#pragma unroll
                for (int s = 0; s < 7; ++s) w[s] = __float2int_rn(acc[s][e]);
                H[e] = (long long)w[0] * h0 + (long long)w[1] * h1 + (long long)w[2] * h2;
                Lw[e] = (long long)w[2] * w2 + (long long)w[3] * w3 + (long long)w[4] * w4 + (long long)w[5] * w5 +
                        (long long)w[6] * w6;
            }
            const int l = lk + gr + (odd ? 8 : 0);
            const double cl = W.c[l - c0], f = (((l & q4) & 1) ? -cl : cl) * sc;     // (-1)^l for P[1]
            double v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const long long h = (odd ? H[2 + e] : H[e]) + __shfl_xor_sync(0xffffffffu, odd ? H[e] : H[2 + e], 2);
                const long long w = (odd ? Lw[2 + e] : Lw[e]) + __shfl_xor_sync(0xffffffffu, odd ? Lw[e] : Lw[2 + e], 2);
                v[e] = f * fma((double)w, 0x1p-36, (double)h);
            }
            if (l <= a.L && (v[0] != 0.0 || v[1] != 0.0)) af_add(a, m, k, l, q4 & 1, v[0], v[1]);
        }
    }
}

// Units in order of m, claimed from *counter by the resident warps (counter null: one per warp).
__global__ void __launch_bounds__(32 * kAfWarps, 4) k_lcontract_adj_fx(const __grid_constant__ AfArgs a, int groups,
                                                                       unsigned nunits, unsigned *counter) {
    extern __shared__ __align__(16) unsigned char af_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    AfWarp &W = reinterpret_cast<AfWarp *>(af_smem)[warp];
    unsigned u = blockIdx.x * kAfWarps + warp;
    if (counter) {
        if (lane == 0) u = atomicAdd(counter, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
    }
    while (u < nunits) {
        unsigned next = 0xffffffffu;
        if (counter && lane == 0) next = atomicAdd(counter, 1u);
        af_unit(a, W, groups, u);
        __syncwarp();
        u = __shfl_sync(0xffffffffu, next, 0);
    }
}

sl_status launch_lcontract_adj_fx(sl_plan *p) {
    AfArgs a;
    a.L = p->L;
    a.K = p->K;
    a.R = p->R;
    a.npairs = p->npairs;
    a.nalm = p->nalm;
    a.xr = p->d_xr;
    a.ls = p->d_ls_adj;
    a.st64 = p->d_st64_adj;
    a.tab = p->d_tab64;
    a.Ghat = p->d_Gadj;
    a.Abar = p->d_Abar;
    const size_t sm = kAfWarps * sizeof(AfWarp);
    cudaError_t e = allow_dyn_smem(k_lcontract_adj_fx, sm);
    if (e != cudaSuccess) return cuda_check(e, "k_lcontract_adj_fx smem attribute");
    // two groups per warp where that leaves several warps for every slot
    int nsm = 152;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
    const int64_t mk = (int64_t)(p->L + 1) * (p->K + 1), slots = (int64_t)nsm * 4 * kAfWarps;
    const int groups = mk * ((p->npairs + 31) / 32) >= 4 * slots ? 2 : 1;
    const int64_t nunits = mk * ((p->npairs + 16 * groups - 1) / (16 * groups));
    if (nunits > 0x7fffffff) return set_error(SL_ERR_UNSUPPORTED, "grid too large");
    unsigned *counter = nullptr;
    if (nunits > slots) {
        counter = p->d_lc_counter;
        if ((e = cudaMemsetAsync(counter, 0, sizeof(unsigned), p->stream)) != cudaSuccess) return cuda_check(e, "unit counter");
    }
    const unsigned nblk = (unsigned)((std::min(nunits, slots) + kAfWarps - 1) / kAfWarps);
    const int slot = timing_begin(p, "lcontract_adj_fx");
    k_lcontract_adj_fx<<<nblk, 32 * kAfWarps, sm, p->stream>>>(a, groups, (unsigned)nunits, counter);
    timing_end(p, slot);
    return cuda_check(cudaGetLastError(), "k_lcontract_adj_fx launch");
}

}  // namespace sl
