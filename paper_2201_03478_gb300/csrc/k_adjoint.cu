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
// from the same FP64 start states (the evanescent zone is skipped).
// computed by k_lcontract_adj_fx (k_adjoint_fx.cu).
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
__global__ void k_grad_sky(int L, int K, int64_t nalm, const double2 *__restrict__ beam,
                           const double2 *__restrict__ Abar, double2 *__restrict__ out, int accumulate) {
    const int m = blockIdx.y, X = blockIdx.z;
    const int l = m + blockIdx.x * blockDim.x + threadIdx.x;
    if (l > L) return;
    const int64_t row = L + 1;
    double2 g = {0.0, 0.0};
    const double sgn = (m & 1) ? -1.0 : 1.0;
    for (int k = 0; k <= K; ++k) {
        double2 b = beam[((int64_t)X * (K + 1) + k) * (L + 1) + l];
        if (k == 0) b.y = 0.0;
        const double2 ap = Abar[((int64_t)k * (2 * L + 1) + L + m) * row + l];
        // b * Abar_{+m}
        g.x += b.x * ap.x - b.y * ap.y;
        g.y += b.x * ap.y + b.y * ap.x;
        if (m > 0) {
            const double2 an = Abar[((int64_t)k * (2 * L + 1) + L - m) * row + l];
            // (-1)^m conj(b) conj(an) = (-1)^m conj(b * an)
            g.x += sgn * (b.x * an.x - b.y * an.y);
            g.y -= sgn * (b.x * an.y + b.y * an.x);
        }
    }
    if (m == 0) g.y = 0.0;
    double2 *o = out + (int64_t)X * nalm + (int64_t)m * (2 * L + 1 - m) / 2 + l;
    if (accumulate) {
        const double2 c = *o;
        g.x += c.x;
        g.y += c.y;
    }
    *o = g;
}

__global__ void k_grad_beam(int L, int K, int64_t nalm, const double2 *__restrict__ sky,
                            const double2 *__restrict__ Abar, double2 *__restrict__ out, int accumulate) {
    const int k = blockIdx.y, X = blockIdx.z;
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l > L) return;
    const int64_t row = L + 1;
    double2 g = {0.0, 0.0};
    if (l >= k) {
        const double2 *Ak = Abar + (int64_t)k * (2 * L + 1) * row;
        for (int m = 0; m <= l; ++m) {
            double2 s = sky[(int64_t)X * nalm + (int64_t)m * (2 * L + 1 - m) / 2 + l];
            if (m == 0) s.y = 0.0;
            const double2 ap = Ak[(int64_t)(L + m) * row + l];
            // s * conj(ap)
            g.x += s.x * ap.x + s.y * ap.y;
            g.y += s.y * ap.x - s.x * ap.y;
            if (m > 0) {
                const double2 an = Ak[(int64_t)(L - m) * row + l];
                const double sg = (m & 1) ? -1.0 : 1.0;
                // (-1)^m conj(s) conj(an) = (-1)^m conj(s * an)
                g.x += sg * (s.x * an.x - s.y * an.y);
                g.y -= sg * (s.x * an.y + s.y * an.x);
            }
        }
        if (k == 0) g.y = 0.0;
    }
    double2 *o = out + ((int64_t)X * (K + 1) + k) * (L + 1) + l;
    if (accumulate) {
        const double2 c = *o;
        g.x += c.x;
        g.y += c.y;
    }
    *o = g;
}

sl_status launch_grad(sl_plan *p, const double *sky, const double *beam, double *sky_grad, double *beam_grad,
                      int accumulate) {
    const int bs = 128;
    if (sky_grad) {
        dim3 grid((p->L + 1 + bs - 1) / bs, p->L + 1, p->ncomp);
        int slot = timing_begin(p, "grad_sky");
        k_grad_sky<<<grid, bs, 0, p->stream>>>(p->L, p->K, p->nalm, (const double2 *)beam, p->d_Abar,
                                              (double2 *)sky_grad, accumulate);
        timing_end(p, slot);
        sl_status st = cuda_check(cudaGetLastError(), "k_grad_sky launch");
        if (st != SL_OK) return st;
    }
    if (beam_grad) {
        dim3 grid((p->L + 1 + bs - 1) / bs, p->K + 1, p->ncomp);
        int slot = timing_begin(p, "grad_beam");
        k_grad_beam<<<grid, bs, 0, p->stream>>>(p->L, p->K, p->nalm, (const double2 *)sky, p->d_Abar,
                                               (double2 *)beam_grad, accumulate);
        timing_end(p, slot);
        return cuda_check(cudaGetLastError(), "k_grad_beam launch");
    }
    return SL_OK;
}

}  // namespace sl
