// LSQR-based SPIR (Sec. 4.2, "SPIR: conjugate gradient or LSQR?"): each
// refinement step's least-squares problem min || r_i - B dy ||, with
// B = A D^{-1} R^{-1} (column scaling and the sketch's R as a right
// preconditioner, eq. (ls-itref)), solved by LSQR (Paige and Saunders) from
// dy = 0, with SPIR's two stopping rules applied to the LSQR step
// (phi_k / rho_k) w_k.
//
// Golub-Kahan bidiagonalisation needs B v and B^T u per iteration.  Both come
// from ONE pass over A: with q_{k+1} = B v_k - alpha_k u_k (unnormalised,
// u_k = q_k / beta_k), the row i of q_{k+1} is (a_i . z) - (alpha_k /
// beta_k) q_k[i] with z = D^{-1} R^{-1} v_k, and row i's share of
// A^T q_{k+1} is a_i q_{k+1}[i] -- known as soon as the row's q is.  So the
// pass is shaped like the residual pass: the m-vector s holds -q_k, the pass
// computes r = bscale s - A z (= -q_{k+1}, with bscale = alpha_k / beta_k in
// the sign convention below), writes it back to s, and sums A^T r and
// ||r||^2 = beta_{k+1}^2.  The n-vector recurrences run in k_inner.cu's
// kernels (method 2).
//
// Sign convention: s starts as r_i = q_1 (written by the step's FP64
// residual pass), so the first pass takes bscale = +alpha_1 / beta_1; every
// pass leaves s = -q_{k+1}, so later passes take bscale = -alpha_k / beta_k.
// R^{-T} D^{-1} A^T s is then -B^T q_{k+1}.
//
// Two forms of the pass: launch_pass_lsqr_df (k_pass_df.cu), on the hi / lo
// FP32 planes of A in double-float (the default, as the inner passes of FOSSILS and SPIR),
// and the FP64 residual pass of k_pass.cu with bscale and s (two FP64 FMAs per
// element; inner_fp64_fma = 1 or planes out of range).
#include "lsq_common.cuh"

namespace lsq {

namespace {

// LSQR start (Paige and Saunders' initialisation) from the step's right-hand
// side: beta_1 u_1 = r_i (kept in s by the residual pass), c = R^{-T} D^{-1}
// A^T r_i = beta_1 B^T u_1, so alpha_1 = ||c|| / beta_1, v_1 = c / ||c||,
// w_1 = v_1, phibar = beta_1, rhobar = alpha_1, dy = 0.
__global__ void __launch_bounds__(kVecThreads)
    lsqr_init_kernel(int n, const double *__restrict__ c, int step, double *v, double *w,
                     double *dy, int max_iters, int use_thresh, DevState *st) {
  const double beta = sqrt(st->r2);
  const double cn = sqrt(st->cnorm2[step]);
  const bool live = beta > 0.0 && cn > 0.0;
  const double inv = live ? 1.0 / cn : 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double vi = c[i] * inv;
    v[i] = vi;
    w[i] = vi;
    dy[i] = 0.0;
  }
  if (threadIdx.x == 0) {
    const double alpha = live ? cn / beta : 0.0;
    st->lq_phibar[0] = beta;
    st->lq_rhobar[0] = alpha;
    st->lq_bscale = live ? alpha / beta : 0.0;
    st->iters = 0;
    st->max_iters = max_iters;
    st->use_thresh = use_thresh;
    st->dnorm2 = 0.0;
    st->done = (max_iters <= 0 || !live) ? 1 : 0;
  }
}

}  // namespace

cudaError_t launch_lsqr_init(int n, const double *c, int step, double *v, double *w, double *dy,
                             int max_iters, int use_thresh, DevState *st, cudaStream_t s) {
  lsqr_init_kernel<<<1, kVecThreads, 0, s>>>(n, c, step, v, w, dy, max_iters, use_thresh, st);
  return cudaGetLastError();
}

}  // namespace lsq
