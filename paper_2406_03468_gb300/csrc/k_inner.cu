// The small kernels of an inner iteration of the refinement loop (Alg. 1's
// Apply around the pass over A, then Polyak's, CG's or LSQR's update):
//
//   pass over A -> reduce_kernel (k_pass.cu): h = D^-1 A^T (A z)
//               -> inner_w_kernel:  w = R^-T h, the update's first half
//               -> inner_u_kernel:  its second half, z = D^-1 R^-1 (next vector)
//
// The two triangular solves are products with X = R^-1, formed once per
// factorisation (tri_inv_kernel, columns by back substitution).  A
// substitution is a chain of n dependent steps, each one FP64 operation
// (67 cycles on GB300) and a shuffle: 39 us per solve at n = 500 on a cluster
// of 8 CTAs (11 us at n = 97, 78 us at n = 1000), two per iteration.  A
// product has no chain: one warp per entry, all SMs: 3 us at n = 128, 4.5 at
// n = 500, 6 - 10 at n = 1000 (bound by latency: the previous kernel's end, one
// L2 round trip, n / 32 products and a warp reduction).  From the end of a
// pass to the start of the next: 14 us at n = 500 (114 before, with the
// vector updates on one CTA), 8 us at n = 128 (54).  Every column of X has a componentwise small residual, R X = I + F
// with |F| <= c u |R| |X|, so the operator of the inner iteration becomes
// (I + F)^T M (I + F): a relative perturbation of the size u kappa that the
// substitutions make too.  The right-hand side c = R^-T g, x0 and the updates
// of x keep back substitution (k_tri.cu).
//
// All four launches of an iteration are programmatic dependents of each
// other: a kernel's CTAs take their slots and load what does not change
// between iterations (the rows of X, D^-1) while the previous kernel ends, and
// wait for its results with griddepcontrol.wait.
//
// The stop decision is taken on the device.  inner_u_kernel's last CTA sets
// DevState::done while others of the launch may not have started, so W and U
// test DevState::ugate, the copy of `done` that the reduction before them
// makes.  Scalars that U's CTAs read and its last CTA replaces are kept twice
// and alternate with the parity of the iteration.
#include "lsq_common.cuh"
#include "lsq_dev.cuh"

namespace lsq {

namespace {

constexpr int kInvCols = 4;         // columns of X per CTA of tri_inv_kernel
constexpr int kInvThreads = 256;
constexpr int kInWarps = 4;         // W and U: one warp per entry, one per sub-partition
constexpr int kInThreads = 32 * kInWarps;

// X = R^-1, kInvCols columns per CTA by blocked back substitution (32 x 32
// blocks, last block row first): the 8 warps share the columns k of
// sum_k R_rk X_kc beyond the block (lane = row r, so R is read coalesced and
// each R_rk serves the 4 columns), then 4 warps run the block's chain, one
// column each, on the tile pre-scaled by 1 / R_ll.  Bound by FP64 work in
// the last columns' CTAs (4 n^2 / 2 FMA on one SM: about 0.15 ms at n = 500,
// 0.6 ms at n = 1000), which start first; it runs beside the first
// residual pass.  X is written in both layouts, zeros below the diagonal
// only inside the diagonal blocks (nothing reads below it).
__device__ __forceinline__ void tri_inv_body(const double *__restrict__ Rcm,
                                             const double *__restrict__ rinv,
                                             const double *__restrict__ Dt, int n,
                                             double *__restrict__ Xcm, double *__restrict__ Xrm,
                                             int cta, double *ism) {
  const int nb = (n + 31) / 32, ldx = 32 * nb;
  double *xs = ism;                          // kInvCols x ldx: the columns so far
  double *red = ism + kInvCols * ldx;        // 8 x kInvCols x 32 partial sums
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j0 = ((n + kInvCols - 1) / kInvCols - 1 - cta) * kInvCols;
  const int jl = min(n, j0 + kInvCols) - 1;  // last column of this CTA
  for (int I = jl / 32; I >= 0; I--) {
    const int r = 32 * I + lane;
    const bool in = r < n;
    double dreg[32], rl = 0.0;
    if (warp < kInvCols) {
      const double *D = Dt + (size_t)I * 1024;
#pragma unroll
      for (int q = 0; q < 32; q++) dreg[q] = D[q * 32 + lane];
      rl = in ? rinv[r] : 0.0;
    }
    double acc[kInvCols];
#pragma unroll
    for (int c = 0; c < kInvCols; c++) acc[c] = 0.0;
#pragma unroll 4
    for (int k = 32 * (I + 1) + warp; k <= jl; k += kInvThreads / 32) {
      const double a = in ? Rcm[(size_t)k * n + r] : 0.0;
#pragma unroll
      for (int c = 0; c < kInvCols; c++) acc[c] = fma(a, xs[c * ldx + k], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < kInvCols; c++) red[(warp * kInvCols + c) * 32 + lane] = acc[c];
    __syncthreads();
    if (warp < kInvCols) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < kInvThreads / 32; w++) s += red[(w * kInvCols + warp) * 32 + lane];
      const int j = j0 + warp;
      s = (((in && r == j) ? 1.0 : 0.0) - s) * rl;
#pragma unroll
      for (int q = 31; q >= 0; q--) {
        const double xq = __shfl_sync(0xffffffffu, s, q);
        if (lane < q) s = fma(-dreg[q], xq, s);
      }
      xs[warp * ldx + r] = s;
      if (in && j < n) {
        Xcm[(size_t)j * n + r] = s;
        Xrm[(size_t)r * n + j] = s;
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kInvThreads)
    tri_inv_kernel(const double *__restrict__ Rcm, const double *__restrict__ rinv,
                   const double *__restrict__ Dt, int n, double *__restrict__ Xcm,
                   double *__restrict__ Xrm) {
  extern __shared__ double ism[];
  tri_inv_body(Rcm, rinv, Dt, n, Xcm, Xrm, blockIdx.x, ism);
}

// Sum over the CTA of kInWarps warps, for every thread.
__device__ __forceinline__ double in_sum(double v, double *scratch) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
  __syncthreads();
  return (scratch[0] + scratch[1]) + (scratch[2] + scratch[3]);
}

// w = X^T h, one warp per entry (a column of X), and per method:
//   0 Polyak:  Delta = alpha (c - w) + beta (dy - dy_old), (dy, dy_old) <-
//              (dy + Delta, dy); the CTA's share of ||Delta||^2 in pn
//   1 CG:      w kept; the CTA's share of p . w in pn
//   2 LSQR:    w <- -w / beta - beta v (beta^2 = lq_b2); its share of the norm
// Latency: the column of X is loaded before the dependency wait, then h.
template <int NB, int METHOD>
__device__ __forceinline__ void inner_w_body(int n, const double *__restrict__ Xcm,
                                             const double *h, double *w, const double *c,
                                             double *dy, double *dyold, const double *pv,
                                             double *pn, const DevState *st, double *scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * kInWarps + warp;
  double xr[NB];
#pragma unroll
  for (int k = 0; k < NB; k++) {
    const int i = 32 * k + lane;
    xr[k] = (j < n && i <= j) ? ld_early(Xcm + (size_t)j * n + i) : 0.0;
  }
  griddep_wait();
  if (*(volatile const int *)&st->ugate) return;
  // the update's operands, on their way during the product
  double e0 = 0.0, e1 = 0.0, e2 = 0.0, e3 = 0.0, e4 = 0.0;
  if (lane == 0 && j < n) {
    if (METHOD == 0) {
      e0 = c[j];
      e1 = dy[j];
      e2 = dyold[j];
      e3 = st->alpha;
      e4 = st->beta;
    } else {
      e0 = pv[j];
      if (METHOD == 2) {
        e1 = sqrt(st->lq_b2);
        e2 = e1 > 0.0 ? 1.0 / e1 : 0.0;
      }
    }
  }
  double hv[NB];  // all loads before the first product: one L2 latency
#pragma unroll
  for (int k = 0; k < NB; k++) {
    const int i = 32 * k + lane;
    hv[k] = (j < n && i <= j) ? h[i] : 0.0;
  }
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    if (32 * k <= j) {  // the warp's column ends at row j
      if (k & 1) a1 = fma(xr[k], hv[k], a1);
      else a0 = fma(xr[k], hv[k], a0);
    }
  }
  const double t = warp_sum(a0 + a1);
  double s = 0.0;
  if (lane == 0 && j < n) {
    if (METHOD == 0) {
      const double delta = e3 * (e0 - t) + e4 * (e1 - e2);
      dyold[j] = e1;
      dy[j] = e1 + delta;
      s = delta * delta;
    } else if (METHOD == 1) {
      w[j] = t;
      s = e0 * t;
    } else {
      const double vi = -t * e2 - e1 * e0;  // beta, 1 / beta
      w[j] = vi;
      s = vi * vi;
    }
  }
  if (lane == 0) scratch[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) pn[blockIdx.x] = (scratch[0] + scratch[1]) + (scratch[2] + scratch[3]);
}

template <int NB, int METHOD>
__global__ void __launch_bounds__(kInThreads)
    inner_w_kernel(int n, const double *__restrict__ Xcm, const double *h, double *w,
                   const double *c, double *dy, double *dyold, const double *pv, double *pn,
                   const DevState *st) {
  griddep_launch();
  __shared__ double scratch[kInWarps];
  inner_w_body<NB, METHOD>(n, Xcm, h, w, c, dy, dyold, pv, pn, st, scratch);
}

__device__ __forceinline__ void u_finish(DevState *st, double dn2, bool exhausted, int *hprog) {
  const int it = st->iters + 1;
  st->iters = it;
  st->dnorm2 = dn2;
  bool stop = it >= st->max_iters || exhausted;
  if (st->use_thresh && sqrt(dn2) <= st->thresh1) stop = true;
  if (stop) st->done = 1;
  // the host's view of the progress (page-locked host memory)
  if (hprog != nullptr) *(volatile int *)hprog = it | (stop ? kProgDone : 0);
}

// z = D^-1 X v, one warp per entry (a row of X), after the update's second
// half; the last CTA has no entries and takes the stop decision.
//   METHOD 0:  v = dy (updated by inner_w_kernel)
//   METHOD 1:  gam = rho / p.q, r <- r - gam q, bet = r.r / rho, v = p <- r + bet p
//              (formed by every CTA in shared memory: 6 FP64 instructions per
//              thread at n = 256 cost less than a launch), dy += gam p
//   METHOD 2:  the plane rotation; v <- vt / alpha, dy += (phi / rho) w,
//              w <- v - (theta / rho) w
//   METHOD 3:  v = src only (the step's first z; no update, no gate)
// Entry i of the vectors is written by the warp of row i alone; what every
// CTA reads (r, p) alternates between two buffers.
// np: the CTAs (partial sums) of inner_w_kernel, and the index of the last one here
template <int NB, int METHOD>
__device__ __forceinline__ void inner_u_body(int n, int np, const double *__restrict__ Xrm,
                                             const double *__restrict__ dinv, const double *src,
                                             double *z, const double *res, double *res_out,
                                             const double *pv, double *pv_out, double *dy,
                                             const double *pn, int par, DevState *st, int *hprog,
                                             double *scratch, double *sv) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * kInWarps + warp;
  const bool fin = METHOD != 3 && (int)blockIdx.x == np;
  double xr[NB], di = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    const int j = 32 * k + lane;
    xr[k] = (i < n && j >= i && j < n) ? ld_early(Xrm + (size_t)i * n + j) : 0.0;
  }
  if (i < n) di = ld_early(dinv + i);
  if (METHOD != 3) {
    griddep_wait();
    // not earlier: the next pass's CTAs would fill the slots of the SMs that
    // finished the last pass first, and run unevenly spread
    griddep_launch();
    if (*(volatile const int *)&st->ugate) return;
  }
  double vv[NB];  // all loads before the first product: one L2 latency
  if (METHOD != 1) {
#pragma unroll
    for (int k = 0; k < NB; k++) {
      const int j = 32 * k + lane;
      vv[k] = (i < n && j >= i && j < n) ? src[j] : 0.0;
    }
  }
  double sum = 0.0;  // METHOD 0: ||Delta||^2, 1: p.q, 2: ||vt||^2
  if (METHOD == 1 || METHOD == 2 || (METHOD == 0 && fin)) {
    double s = 0.0;
    for (int q = threadIdx.x; q < np; q += kInThreads) s += pn[q];
    sum = in_sum(s, scratch);
  }
  if (METHOD == 0 && fin) {
    if (threadIdx.x == 0) u_finish(st, sum, false, hprog);
    return;
  }
  double gam = 0.0;
  if (METHOD == 1) {
    const double rho = st->rho_ab[par];
    gam = rho / sum;
    double rr = 0.0, ss = 0.0;
    for (int q = threadIdx.x; q < n; q += kInThreads) {
      const double r = res[q] - gam * src[q];
      sv[q] = r;
      rr = fma(r, r, rr);
      if (fin) {
        const double step = gam * pv[q];
        ss = fma(step, step, ss);
      }
    }
    rr = in_sum(rr, scratch);
    if (fin) {
      ss = in_sum(ss, scratch);
      if (threadIdx.x == 0) {
        st->rho_ab[par ^ 1] = rr;
        u_finish(st, ss, !(rr > 0.0), hprog);
      }
      return;
    }
    const double bet = rr / rho;
    for (int q = threadIdx.x; q < n; q += kInThreads) sv[q] = sv[q] + bet * pv[q];
    __syncthreads();
  }
  double ia = 1.0, tstep = 0.0, tw = 0.0;
  if (METHOD == 2) {
    const double beta = sqrt(st->lq_b2);
    const double alpha = sqrt(sum);
    ia = alpha > 0.0 ? 1.0 / alpha : 0.0;
    const double rhobar = st->lq_rhobar[par], phibar = st->lq_phibar[par];
    const double rho = hypot(rhobar, beta);
    const double cs = rhobar / rho, sn = beta / rho;
    const double theta = sn * alpha, phi = cs * phibar;
    tstep = phi / rho;
    tw = theta / rho;
    if (fin) {
      double ss = 0.0;
      for (int q = threadIdx.x; q < n; q += kInThreads) {
        const double step = tstep * res[q];
        ss = fma(step, step, ss);
      }
      ss = in_sum(ss, scratch);
      if (threadIdx.x == 0) {
        st->lq_rhobar[par ^ 1] = -cs * alpha;
        st->lq_phibar[par ^ 1] = sn * phibar;
        st->lq_bscale = beta > 0.0 ? -alpha / beta : 0.0;
        u_finish(st, ss, !(alpha > 0.0) || !(sn * phibar != 0.0), hprog);
      }
      return;
    }
  }
  if (METHOD == 1) {
#pragma unroll
    for (int k = 0; k < NB; k++) {
      const int j = 32 * k + lane;
      vv[k] = (i < n && j >= i && j < n) ? sv[j] : 0.0;
    }
  }
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    if (32 * k + 31 >= i) {  // the warp's row starts at column i
      if (k & 1) a1 = fma(xr[k], vv[k], a1);
      else a0 = fma(xr[k], vv[k], a0);
    }
  }
  const double t = warp_sum(a0 + a1);
  if (lane == 0 && i < n) {
    z[i] = di * (METHOD == 2 ? t * ia : t);
    if (METHOD == 1) {
      const double p = pv[i];
      res_out[i] = res[i] - gam * src[i];
      pv_out[i] = sv[i];
      dy[i] += gam * p;
    } else if (METHOD == 2) {
      // LSQR's w alternates like r; its v (pv_out) is read by no CTA here
      const double vi = src[i] * ia, wi = res[i];
      pv_out[i] = vi;
      dy[i] += tstep * wi;
      res_out[i] = vi - tw * wi;
    }
  }
}

template <int NB, int METHOD>
__global__ void __launch_bounds__(kInThreads)
    inner_u_kernel(int n, const double *__restrict__ Xrm, const double *__restrict__ dinv,
                   const double *src, double *z, const double *res, double *res_out,
                   const double *pv, double *pv_out, double *dy, const double *pn, int par,
                   DevState *st, int *hprog) {
  __shared__ double scratch[kInWarps];
  __shared__ double sv[METHOD == 1 ? 32 * NB : 1];
  inner_u_body<NB, METHOD>(n, gridDim.x - 1, Xrm, dinv, src, z, res, res_out, pv, pv_out, dy, pn,
                           par, st, hprog, scratch, sv);
}

// One step of both condition-estimate chains (blockIdx.y): out = M (v / ||v||)
// with one warp per entry and the CTAs' shares of ||out||^2.
//   chain 0, sigma_max(R):     M = R, R^T, R, ... (power iteration on R^T R)
//   chain 1, 1 / sigma_min(R): M = X^T, X, X^T, ... with X = R^-1
// Step 0 takes the fixed start vectors.  A step is a latency of about 3 us
// (21 steps: one CTA with substitutions took 0.8 ms at n = 97, 2.9 at 500 and
// 7.6 at 1000).
__device__ __forceinline__ double cond_start(int chain, int i) {
  return 1.0 + 0.25 * (double)(chain == 0 ? (i * 7919) % 17 : (i * 104729) % 13);
}

template <int NB>
__device__ __forceinline__ void cond_step_body(int n, int np, const double *__restrict__ Rcm,
                                               const double *__restrict__ Rrm,
                                               const double *__restrict__ Xcm,
                                               const double *__restrict__ Xrm, int step,
                                               const double *vin, const double *pin, double *vout,
                                               double *pout, double *scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, chain = blockIdx.y;
  const int i = blockIdx.x * kInWarps + warp;
  const bool upper = ((step & 1) ^ chain) == 0;  // row i of R or X, else column i
  const double *M = chain == 0 ? (upper ? Rrm : Rcm) : (upper ? Xrm : Xcm);
  double mr[NB], vv[NB];
#pragma unroll
  for (int k = 0; k < NB; k++) {
    const int j = 32 * k + lane;
    const bool in = i < n && j < n && (upper ? j >= i : j <= i);
    mr[k] = in ? ld_early(M + (size_t)i * n + j) : 0.0;
  }
  griddep_wait();
  vin += (size_t)chain * n;
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    const int j = 32 * k + lane;
    const bool in = i < n && j < n && (upper ? j >= i : j <= i);
    vv[k] = !in ? 0.0 : step == 0 ? cond_start(chain, j) : vin[j];
  }
  if (step == 0) {
    for (int j = threadIdx.x; j < n; j += kInThreads) s = fma(cond_start(chain, j), cond_start(chain, j), s);
  } else {
    for (int q = threadIdx.x; q < np; q += kInThreads) s += pin[chain * np + q];
  }
  s = sqrt(in_sum(s, scratch));
  const double inv = s > 0.0 ? 1.0 / s : 0.0;
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    if (upper ? 32 * k + 31 >= i : 32 * k <= i) {
      if (k & 1) a1 = fma(mr[k], vv[k], a1);
      else a0 = fma(mr[k], vv[k], a0);
    }
  }
  const double t = warp_sum(a0 + a1) * inv;
  if (lane == 0 && i < n) vout[(size_t)chain * n + i] = t;
  __syncthreads();
  if (lane == 0) scratch[warp] = i < n ? t * t : 0.0;
  __syncthreads();
  if (threadIdx.x == 0)
    pout[chain * np + blockIdx.x] = (scratch[0] + scratch[1]) + (scratch[2] + scratch[3]);
}

template <int NB>
__global__ void __launch_bounds__(kInThreads)
    cond_step_kernel(int n, const double *__restrict__ Rcm, const double *__restrict__ Rrm,
                     const double *__restrict__ Xcm, const double *__restrict__ Xrm, int step,
                     const double *vin, const double *pin, double *vout, double *pout) {
  griddep_launch();
  __shared__ double scratch[kInWarps];
  cond_step_body<NB>(n, gridDim.x, Rcm, Rrm, Xcm, Xrm, step, vin, pin, vout, pout, scratch);
}

__device__ __forceinline__ void cond_finish_body(const double *pin, int np, DevState *st,
                                                 double *scratch) {
  double s0 = 0.0, s1 = 0.0;
  for (int q = threadIdx.x; q < np; q += kInThreads) {
    s0 += pin[q];
    s1 += pin[np + q];
  }
  s0 = in_sum(s0, scratch);
  s1 = in_sum(s1, scratch);
  if (threadIdx.x == 0) {
    const double smax = sqrt(s0), winv = sqrt(s1);
    const double smin = (winv > 0.0) ? 1.0 / winv : 0.0;
    st->normest = smax;
    st->condest = (smin > 0.0) ? smax / smin : INFINITY;
  }
}

__global__ void __launch_bounds__(kInThreads)
    cond_finish_kernel(const double *pin, int np, DevState *st) {
  griddep_wait();
  __shared__ double scratch[kInWarps];
  cond_finish_body(pin, np, st, scratch);
}

// Step-2 count: q0 of Theorem 7.1 with kappa := condest and distortion
// 1.01 eta; Alg. 5 returns dy_(q) after q - 1 updates (as the plan path).
__device__ int step2_count(double condest, double eta, int max_inner) {
  const double e = 1.01 * eta;
  double q0 = 11.0;
  if (e > 0.0 && isfinite(condest) && condest > 0.0) {
    const double v = 1.0 + 2.0 * log(1.0 / (condest * kU)) / log(1.0 / e);
    q0 = v > 11.0 ? v : 11.0;
  }
  int q = (int)ceil(q0) - 1;
  if (q < 1) q = 1;
  if (q > max_inner) q = max_inner;
  return q;
}

// ---------------------------------------------------------------------------
// The same kernels for the items of a batch (lsq_batch.cu): blockIdx.z is the
// item.  Ordinary launches inside captured graphs; a CTA beyond its item's
// entries returns.
// ---------------------------------------------------------------------------

// Buffers and partial sums of a condition-estimate step in the item's cw.
__device__ __forceinline__ void b_cond_bufs(const BItem &it, int np, int step, const double *&vi,
                                            const double *&pi, double *&vo, double *&po) {
  double *v = it.cw, *p = it.cw + 4 * (size_t)it.n;
  vi = v + (step & 1) * 2 * (size_t)it.n;
  vo = v + ((step & 1) ^ 1) * 2 * (size_t)it.n;
  pi = p + (step & 1) * 2 * (size_t)np;
  po = p + ((step & 1) ^ 1) * 2 * (size_t)np;
}

__global__ void __launch_bounds__(kInvThreads) b_tri_inv_kernel(const BItem *__restrict__ items) {
  extern __shared__ double ism[];
  const BItem &it = items[blockIdx.z];
  if ((int)blockIdx.x * kInvCols >= it.n) return;
  tri_inv_body(it.Rcm, it.rinv, it.Dt, it.n, it.Xcm, it.Xrm, blockIdx.x, ism);
}

template <int NB>
__global__ void __launch_bounds__(kInThreads)
    b_cond_step_kernel(const BItem *__restrict__ items, int step) {
  __shared__ double scratch[kInWarps];
  const BItem &it = items[blockIdx.z];
  const int np = (it.n + kInWarps - 1) / kInWarps;
  if ((int)blockIdx.x >= np) return;
  const double *vi, *pi;
  double *vo, *po;
  b_cond_bufs(it, np, step, vi, pi, vo, po);
  cond_step_body<NB>(it.n, np, it.Rcm, it.Rrm, it.Xcm, it.Xrm, step, vi, pi, vo, po, scratch);
}

// condest / normest and the step-2 count (Theorem 7.1 with kappa := condest)
__global__ void __launch_bounds__(kInThreads)
    b_cond_finish_kernel(const BItem *__restrict__ items, int last, int max_inner) {
  __shared__ double scratch[kInWarps];
  const BItem &it = items[blockIdx.z];
  const int np = (it.n + kInWarps - 1) / kInWarps;
  const double *vi, *pi;
  double *vo, *po;
  b_cond_bufs(it, np, last + 1, vi, pi, vo, po);
  cond_finish_body(pi, np, it.st, scratch);
  if (threadIdx.x == 0) it.st->q2 = step2_count(it.st->condest, it.eta, max_inner);
}

template <int NB>
__global__ void __launch_bounds__(kInThreads) b_inner_w_kernel(const BItem *__restrict__ items) {
  __shared__ double scratch[kInWarps];
  const BItem &it = items[blockIdx.z];
  if ((int)blockIdx.x * kInWarps >= it.n) return;
  if (it.method == 0)
    inner_w_body<NB, 0>(it.n, it.Xcm, it.h, it.w, it.c, it.dy, it.dyold, nullptr, it.pn, it.st,
                        scratch);
  else
    inner_w_body<NB, 1>(it.n, it.Xcm, it.h, it.w, it.c, it.dy, it.dyold,
                        it.st->par ? it.p2 : it.p, it.pn, it.st, scratch);
}

// first = 1: the step's first z
template <int NB>
__global__ void __launch_bounds__(kInThreads)
    b_inner_u_kernel(const BItem *__restrict__ items, int first) {
  __shared__ double scratch[kInWarps];
  __shared__ double sv[32 * NB];
  const BItem &it = items[blockIdx.z];
  const int np = (it.n + kInWarps - 1) / kInWarps;
  if ((int)blockIdx.x > np) return;
  if (first) {
    inner_u_body<NB, 3>(it.n, np, it.Xrm, it.dinv, it.method == 0 ? it.dy : it.p, it.z, nullptr,
                        nullptr, nullptr, nullptr, nullptr, nullptr, 0, it.st, nullptr, scratch,
                        sv);
  } else if (it.method == 0) {
    inner_u_body<NB, 0>(it.n, np, it.Xrm, it.dinv, it.dy, it.z, nullptr, nullptr, nullptr, nullptr,
                        it.dy, it.pn, 0, it.st, nullptr, scratch, sv);
  } else {
    const int par = it.st->par;
    inner_u_body<NB, 1>(it.n, np, it.Xrm, it.dinv, it.w, it.z, par ? it.res2 : it.res,
                        par ? it.res : it.res2, par ? it.p2 : it.p, par ? it.p : it.p2, it.dy,
                        it.pn, par, it.st, nullptr, scratch, sv);
  }
}

// k vectors: one warp per entry i of 8 vectors (row i of X, or column i for X^T,
// loaded once).  n <= 256.  The 8 sums by recursive halving over lanes 16, 8
// and 4 apart, then two butterflies: 9 FP64 additions instead of 40.
template <int NB>
__global__ void __launch_bounds__(kInThreads)
    multi_xprod_kernel(int n, int trans, const double *__restrict__ X, const double *__restrict__ V,
                       const double *__restrict__ os, double *__restrict__ out,
                       const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * kInWarps + warp;
  if (i >= n) return;
  V += (size_t)blockIdx.y * 8 * n;
  double acc[8];
#pragma unroll
  for (int c = 0; c < 8; c++) acc[c] = 0.0;
#pragma unroll
  for (int k = 0; k < NB; k++) {
    if (trans ? 32 * k <= i : 32 * k + 31 >= i) {
      const int j = 32 * k + lane;
      const bool in = j < n && (trans ? j <= i : j >= i);
      const double x = in ? X[(size_t)i * n + j] : 0.0;
#pragma unroll
      for (int c = 0; c < 8; c++) acc[c] = fma(x, in ? V[(size_t)c * n + j] : 0.0, acc[c]);
    }
  }
#pragma unroll
  for (int q = 4, o = 16; q >= 1; q >>= 1, o >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int c = 0; c < q; c++) {
      const double keep = hi ? acc[c + q] : acc[c], send = hi ? acc[c] : acc[c + q];
      acc[c] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double t = acc[0];
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  // lane's vector: 4 (bit 4) + 2 (bit 3) + 1 (bit 2)
  const int c = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
  if ((lane & 3) == 0)
    out[((size_t)blockIdx.y * 8 + c) * n + i] = os != nullptr ? os[i] * t : t;
}

}  // namespace

// columns of 32 rows of X held in registers by a warp: the power of two that
// covers n
#define LSQ_NB_SWITCH(N, ...)                                \
  do {                                                       \
    const int nb_ = ((N) + 31) / 32;                         \
    if (nb_ <= 2) { constexpr int NB = 2; __VA_ARGS__; }     \
    else if (nb_ <= 4) { constexpr int NB = 4; __VA_ARGS__; }   \
    else if (nb_ <= 8) { constexpr int NB = 8; __VA_ARGS__; }   \
    else if (nb_ <= 16) { constexpr int NB = 16; __VA_ARGS__; } \
    else { constexpr int NB = 32; __VA_ARGS__; }             \
  } while (0)

cudaError_t launch_tri_inv(const double *Rcm, const double *rinv, const double *Dt, int n,
                           double *Xcm, double *Xrm, cudaStream_t s) {
  const int nb = (n + 31) / 32;
  const size_t smem = sizeof(double) * (size_t)(kInvCols * 32 * nb + (kInvThreads / 32) * kInvCols * 32);
  tri_inv_kernel<<<(n + kInvCols - 1) / kInvCols, kInvThreads, smem, s>>>(Rcm, rinv, Dt, n, Xcm, Xrm);
  return cudaGetLastError();
}

int inner_partials(int n) { return (n + kInWarps - 1) / kInWarps; }

size_t cond_work(int n) { return 4 * (size_t)n + 4 * (size_t)inner_partials(n); }

cudaError_t launch_condest(const double *Rcm, const double *Rrm, const double *Xcm,
                           const double *Xrm, int n, int iters, double *work, DevState *st,
                           cudaStream_t s) {
  const int np = inner_partials(n);
  double *v[2] = {work, work + 2 * (size_t)n};
  double *p[2] = {work + 4 * (size_t)n, work + 4 * (size_t)n + 2 * (size_t)np};
  const dim3 grid(np, 2);
  LSQ_NB_SWITCH(n, {
    for (int k = 0; k <= 2 * iters; k++) {
      const double *vi = v[k & 1], *pi = p[k & 1];
      double *vo = v[(k & 1) ^ 1], *po = p[(k & 1) ^ 1];
      if (k == 0)  // X was written by the kernel before: an ordinary launch
        cond_step_kernel<NB><<<grid, kInThreads, 0, s>>>(n, Rcm, Rrm, Xcm, Xrm, k, vi, pi, vo, po);
      else if (cudaError_t e = launch_pdl(cond_step_kernel<NB>, grid, dim3(kInThreads), 0, s, n,
                                          Rcm, Rrm, Xcm, Xrm, k, vi, pi, vo, po))
        return e;
    }
  });
  return launch_pdl(cond_finish_kernel, dim3(1), dim3(kInThreads), 0, s,
                    (const double *)p[1], np, st);
}

cudaError_t launch_b_cond(const BItem *items, int count, int nmax, int iters, int max_inner,
                          cudaStream_t s) {
  const int nb = (nmax + 31) / 32;
  const size_t smem =
      sizeof(double) * (size_t)(kInvCols * 32 * nb + (kInvThreads / 32) * kInvCols * 32);
  b_tri_inv_kernel<<<dim3((nmax + kInvCols - 1) / kInvCols, 1, count), kInvThreads, smem, s>>>(items);
  const dim3 grid(inner_partials(nmax), 2, count);
  LSQ_NB_SWITCH(nmax, {
    for (int k = 0; k <= 2 * iters; k++)
      b_cond_step_kernel<NB><<<grid, kInThreads, 0, s>>>(items, k);
  });
  b_cond_finish_kernel<<<dim3(1, 1, count), kInThreads, 0, s>>>(items, 2 * iters, max_inner);
  return cudaGetLastError();
}

cudaError_t launch_b_w(const BItem *items, int count, int nmax, cudaStream_t s) {
  const dim3 grid(inner_partials(nmax), 1, count);
  LSQ_NB_SWITCH(nmax, { b_inner_w_kernel<NB><<<grid, kInThreads, 0, s>>>(items); });
  return cudaGetLastError();
}

cudaError_t launch_b_u(const BItem *items, int count, int nmax, int first, cudaStream_t s) {
  const dim3 grid(inner_partials(nmax) + 1, 1, count);
  LSQ_NB_SWITCH(nmax, { b_inner_u_kernel<NB><<<grid, kInThreads, 0, s>>>(items, first); });
  return cudaGetLastError();
}

cudaError_t launch_inner_w(int method, const InnerVecs &v, int par, cudaStream_t s) {
  const int g = inner_partials(v.n);
  const double *pv = method == 1 ? v.p[par] : v.p[0];
  LSQ_NB_SWITCH(v.n, {
    switch (method) {
      case 0:
        return launch_pdl(inner_w_kernel<NB, 0>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xcm, v.h,
                          v.w, v.c, v.dy, v.dyold, pv, v.pn, (const DevState *)v.st);
      case 1:
        return launch_pdl(inner_w_kernel<NB, 1>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xcm, v.h,
                          v.w, v.c, v.dy, v.dyold, pv, v.pn, (const DevState *)v.st);
      default:
        return launch_pdl(inner_w_kernel<NB, 2>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xcm, v.h,
                          v.w, v.c, v.dy, v.dyold, pv, v.pn, (const DevState *)v.st);
    }
  });
}

cudaError_t launch_inner_u(int method, const InnerVecs &v, int par, cudaStream_t s) {
  const int g = inner_partials(v.n) + 1;
  LSQ_NB_SWITCH(v.n, {
    switch (method) {
      case 0:
        return launch_pdl(inner_u_kernel<NB, 0>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xrm,
                          v.dinv, (const double *)v.dy, v.z, (const double *)nullptr,
                          (double *)nullptr, (const double *)nullptr, (double *)nullptr, v.dy,
                          (const double *)v.pn, par, v.st, v.hprog);
      case 1:
        return launch_pdl(inner_u_kernel<NB, 1>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xrm,
                          v.dinv, (const double *)v.w, v.z, (const double *)v.res[par],
                          v.res[par ^ 1], (const double *)v.p[par], v.p[par ^ 1], v.dy,
                          (const double *)v.pn, par, v.st, v.hprog);
      default:
        return launch_pdl(inner_u_kernel<NB, 2>, dim3(g), dim3(kInThreads), 0, s, v.n, v.Xrm,
                          v.dinv, (const double *)v.w, v.z, (const double *)v.res[par],
                          v.res[par ^ 1], (const double *)nullptr, v.p[0], v.dy,
                          (const double *)v.pn, par, v.st, v.hprog);
    }
  });
}

cudaError_t launch_multi_xprod(int n, int k, int trans, const double *X, const double *V,
                               const double *os, double *out, const DevState *gate,
                               cudaStream_t s) {
  const dim3 grid(inner_partials(n), k / 8);
  if (n > 256) return cudaErrorInvalidValue;
  LSQ_NB_SWITCH(n, {
    multi_xprod_kernel<NB><<<grid, kInThreads, 0, s>>>(n, trans, X, V, os, out, gate);
    return cudaGetLastError();
  });
}

cudaError_t launch_inner_z(int method, const InnerVecs &v, cudaStream_t s) {
  const double *src = method == 0 ? v.dy : v.p[0];
  LSQ_NB_SWITCH(v.n, {
    inner_u_kernel<NB, 3><<<inner_partials(v.n), kInThreads, 0, s>>>(
        v.n, v.Xrm, v.dinv, src, v.z, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0,
        v.st, nullptr);
    return cudaGetLastError();
  });
}

}  // namespace lsq
