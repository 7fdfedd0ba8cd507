// k_adjoint.cu -- transpose of the spin "Legendre" step and the final
// sky x beam products (the gradients of the total convolution, Sect. 2.1,
// with respect to the sky s_lm and the beam b_lk).
//
// Contraction transpose (real inner product Re<x, y>):
//   Abar_{k,l,m} = sum_r d^l_{mk}(theta_r) Ghat_k(r, m),   m in [-L, L].
// With the reflections of the forward step, per north ring pair (d1 = d_{m,+k},
// d2 = d_{m,-k}, s_l = (-1)^l):
//   Abar_{+m}(l) = c_l sum_pairs [y1 Ghat(N,+m) + s_l y2 (-1)^m Ghat(S,+m)]
//   Abar_{-m}(l) = c_l sum_pairs [y2 (-1)^{m+k} Ghat(N,-m) + s_l y1 (-1)^k Ghat(S,-m)]
// where d = c y are the rescaled recurrence values of the forward kernel, run
// from the same FP64 start states (the evanescent zone is skipped), computed by
// k_lcontract_adj_fx (k_adjoint_fx.cu).
//
// Products (A_{k,lm} = sum_X s^X_lm conj(b^X_lk), extended to m < 0 by
// s_{l,-m} = (-1)^m conj(s_lm)); g = d/dRe + i d/dIm:
//   sky,  m > 0: sum_k [b_lk Abar_{k,l,m} + (-1)^m conj(b_lk) conj(Abar_{k,l,-m})]
//   sky,  m = 0: sum_k Re(b_lk Abar_{k,l,0})
//   beam:        sum_{m=-l..l} s_lm conj(Abar_{k,lm})   (Re only for k = 0; 0 for l < k)
#include "sl_internal.cuh"

namespace sl {

sl_status launch_lcontract_adjoint(sl_plan *p) {
    sl_status st = cuda_check(cudaMemsetAsync(p->d_Abar, 0,
                                              (size_t)(p->K + 1) * (2 * p->L + 1) * (p->L + 1) * sizeof(double2),
                                              p->stream),
                              "memset Abar");
    if (st != SL_OK) return st;
    return launch_lcontract_adj_fx(p);
}

// ------------------------------------------------------------------ products
// All NC components of a thread together, so that Abar (0.57 GB at lmax 1024, K = 16) is read once and not
// once per component.  Bound by the FP64 pipe at NC = 3 (0.46 ms of it there): 0.623 -> 0.617 ms.
template <int NC>
__global__ void k_grad_sky(int L, int K, int64_t nalm, const double2 *__restrict__ beam,
                           const double2 *__restrict__ Abar, double2 *__restrict__ out, int accumulate) {
    const int m = blockIdx.y;
    const int l = m + blockIdx.x * blockDim.x + threadIdx.x;
    if (l > L) return;
    const int64_t row = L + 1;
    double2 g[NC];
#pragma unroll
    for (int X = 0; X < NC; ++X) g[X] = make_double2(0.0, 0.0);
    const double sgn = (m & 1) ? -1.0 : 1.0;
    for (int k = 0; k <= K; ++k) {
        const double2 ap = Abar[((int64_t)k * (2 * L + 1) + L + m) * row + l];
        const double2 an = m > 0 ? Abar[((int64_t)k * (2 * L + 1) + L - m) * row + l] : make_double2(0.0, 0.0);
#pragma unroll
        for (int X = 0; X < NC; ++X) {
            double2 b = beam[((int64_t)X * (K + 1) + k) * (L + 1) + l];
            if (k == 0) b.y = 0.0;
            // b * Abar_{+m}
            g[X].x += b.x * ap.x - b.y * ap.y;
            g[X].y += b.x * ap.y + b.y * ap.x;
            if (m > 0) {
                // (-1)^m conj(b) conj(an) = (-1)^m conj(b * an)
                g[X].x += sgn * (b.x * an.x - b.y * an.y);
                g[X].y -= sgn * (b.x * an.y + b.y * an.x);
            }
        }
    }
#pragma unroll
    for (int X = 0; X < NC; ++X) {
        if (m == 0) g[X].y = 0.0;
        double2 *o = out + (int64_t)X * nalm + (int64_t)m * (2 * L + 1 - m) / 2 + l;
        if (accumulate) {
            const double2 c = *o;
            g[X].x += c.x;
            g[X].y += c.y;
        }
        *o = g[X];
    }
}

// 32 l x kGbSlices slices of m (m = slice, slice + kGbSlices, ..) a CTA, the slices' sums added
// in shared memory (one thread a value walked its m alone, on few CTAs): lmax 1024, K = 16, NC = 3
// 1.09 -> 0.91 ms, bound as k_grad_sky; lmax 64, K = 4 53 -> 14 us.
constexpr int kGbSlices = 16;

template <int NC>
__global__ void __launch_bounds__(32 * kGbSlices) k_grad_beam(int L, int K, int64_t nalm,
                                                               const double2 *__restrict__ sky,
                                                               const double2 *__restrict__ Abar,
                                                               double2 *__restrict__ out, int accumulate) {
    __shared__ double2 part[NC][kGbSlices][32];
    const int k = blockIdx.y, l = blockIdx.x * 32 + threadIdx.x;
    const int64_t row = L + 1;
    double2 g[NC];
#pragma unroll
    for (int X = 0; X < NC; ++X) g[X] = make_double2(0.0, 0.0);
    if (l <= L && l >= k) {
        const double2 *Ak = Abar + (int64_t)k * (2 * L + 1) * row;
        for (int m = threadIdx.y; m <= l; m += kGbSlices) {
            const double2 ap = Ak[(int64_t)(L + m) * row + l];
            const double2 an = m > 0 ? Ak[(int64_t)(L - m) * row + l] : make_double2(0.0, 0.0);
            const double sg = (m & 1) ? -1.0 : 1.0;
#pragma unroll
            for (int X = 0; X < NC; ++X) {
                double2 s = sky[(int64_t)X * nalm + (int64_t)m * (2 * L + 1 - m) / 2 + l];
                if (m == 0) s.y = 0.0;
                // s * conj(ap)
                g[X].x += s.x * ap.x + s.y * ap.y;
                g[X].y += s.y * ap.x - s.x * ap.y;
                if (m > 0) {
                    // (-1)^m conj(s) conj(an) = (-1)^m conj(s * an)
                    g[X].x += sg * (s.x * an.x - s.y * an.y);
                    g[X].y -= sg * (s.x * an.y + s.y * an.x);
                }
            }
        }
    }
#pragma unroll
    for (int X = 0; X < NC; ++X) part[X][threadIdx.y][threadIdx.x] = g[X];
    __syncthreads();
    const int X = threadIdx.y;
    if (X >= NC || l > L) return;
    double2 t = part[X][0][threadIdx.x];
    for (int y = 1; y < kGbSlices; ++y) {
        t.x += part[X][y][threadIdx.x].x;
        t.y += part[X][y][threadIdx.x].y;
    }
    if (k == 0) t.y = 0.0;
    double2 *o = out + ((int64_t)X * (K + 1) + k) * (L + 1) + l;
    if (accumulate) {
        const double2 c = *o;
        t.x += c.x;
        t.y += c.y;
    }
    *o = t;
}

sl_status launch_grad(sl_plan *p, const double *sky, const double *beam, double *sky_grad, double *beam_grad,
                      int accumulate) {
    const int bs = 128;
    if (sky_grad) {
        dim3 grid((p->L + 1 + bs - 1) / bs, p->L + 1);
        auto kern = p->ncomp == 1 ? k_grad_sky<1> : k_grad_sky<3>;
        int slot = timing_begin(p, "grad_sky");
        kern<<<grid, bs, 0, p->stream>>>(p->L, p->K, p->nalm, (const double2 *)beam, p->d_Abar,
                                              (double2 *)sky_grad, accumulate);
        timing_end(p, slot);
        sl_status st = cuda_check(cudaGetLastError(), "k_grad_sky launch");
        if (st != SL_OK) return st;
    }
    if (beam_grad) {
        dim3 grid((p->L + 1 + 31) / 32, p->K + 1);
        auto kern = p->ncomp == 1 ? k_grad_beam<1> : k_grad_beam<3>;
        int slot = timing_begin(p, "grad_beam");
        kern<<<grid, dim3(32, kGbSlices), 0, p->stream>>>(p->L, p->K, p->nalm, (const double2 *)sky, p->d_Abar,
                                               (double2 *)beam_grad, accumulate);
        timing_end(p, slot);
        return cuda_check(cudaGetLastError(), "k_grad_beam launch");
    }
    return SL_OK;
}

}  // namespace sl
