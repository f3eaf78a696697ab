// The streaming passes over A itself of the refinement loop (Alg. 1; the
// default inner passes, over the FP32 planes of A, are in k_pass_df.cu):
//   pass_resid:  r = b - A x,  g = A^T r,  ||r||^2       (refinement RHS)
//   pass_atax:   h = A^T (A z)                           (inner operator)
// Each reads A exactly once.  One warp owns one row at a time: 16-byte
// streaming loads (evict-first; A is far larger than L2), the row dot
// product is reduced with warp shuffles, and the same registers then feed
// the A^T update into per-lane column accumulators.  Rows are split into
// contiguous ranges, one per CTA (2 CTAs per SM); each CTA writes one
// partial n-vector and a separate kernel sums the partials in a fixed order,
// so the result does not depend on scheduling.
#include "lsq_common.cuh"
#include "lsq_resid.cuh"

namespace lsq {

namespace {

template <int NC, bool VEC>
__device__ __forceinline__ void load_row(const double *__restrict__ row, int n, int lane,
                                         double (&a)[2 * NC]) {
#pragma unroll
  for (int k = 0; k < NC; k++) {
    const int col = 64 * k + 2 * lane;
    if (VEC && col + 1 < n) {
      const double2 v = __ldcs(reinterpret_cast<const double2 *>(row + col));
      a[2 * k] = v.x;
      a[2 * k + 1] = v.y;
    } else {
      a[2 * k] = (col < n) ? __ldcs(row + col) : 0.0;
      a[2 * k + 1] = (col + 1 < n) ? __ldcs(row + col + 1) : 0.0;
    }
  }
}

template <int NC>
__device__ __forceinline__ void load_vec(const double *__restrict__ x, int n, int lane,
                                         double (&v)[2 * NC]) {
#pragma unroll
  for (int k = 0; k < NC; k++) {
    const int col = 64 * k + 2 * lane;
    v[2 * k] = (col < n) ? x[col] : 0.0;
    v[2 * k + 1] = (col + 1 < n) ? x[col + 1] : 0.0;
  }
}

// Deterministic CTA reduction of the per-lane column accumulators into part[blockIdx.x].
template <int NC>
__device__ __forceinline__ void cta_store_partial(const double (&h)[2 * NC], double *sh,
                                                  double *__restrict__ part, int npad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < NC * 64; i += blockDim.x) sh[i] = 0.0;
  for (int w = 0; w < nw; w++) {
    __syncthreads();
    if (warp == w) {
#pragma unroll
      for (int k = 0; k < NC; k++) {
        sh[64 * k + 2 * lane] += h[2 * k];
        sh[64 * k + 2 * lane + 1] += h[2 * k + 1];
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < npad; i += blockDim.x) part[(size_t)blockIdx.x * npad + i] = sh[i];
}

template <int NC, bool VEC>
__global__ void __launch_bounds__(kPassThreads, NC >= 16 ? 1 : kPassCtasPerSm)
    atax_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int n,
                const double *__restrict__ z, double *__restrict__ part, int npad,
                const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  __shared__ double sh[NC * 64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(m, (int64_t)blockIdx.x * per), r1 = min(m, r0 + per);
  double zr[2 * NC], h[2 * NC];
  load_vec<NC>(z, n, lane, zr);
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) h[k] = 0.0;
  for (int64_t i = r0 + warp; i < r1; i += nw) {
    double a[2 * NC];
    load_row<NC, VEC>(A + i * lda, n, lane, a);
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) t = fma(a[k], zr[k], t);
    t = warp_sum(t);
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) h[k] = fma(a[k], t, h[k]);
  }
  cta_store_partial<NC>(h, sh, part, npad);
}

// ---------------------------------------------------------------------------
// Inner pass with the row dot products on the FP32 pipe.
//
// GB300 runs FP64 at about 2 FMA / clock / SM, so two FP64 FMAs per element
// (t_i += a_ij z_j and h_j += a_ij t_i) cap the pass near 30% of HBM.  Here
// t_i is evaluated exactly enough without FP64 arithmetic:
//   * a_ij (FP64, times 2^-Eg) is split into two FP32 words with integer
//     operations: hi = the leading 24 significant bits (exact), lo = the
//     remaining 29 bits rounded to FP32, so |a - hi - lo| <= 2^-48 |a|;
//   * z_j (times 2^Eg 2^-Fz, Fz from max |z'|) is split hi/lo by rounding;
//   * products hi*hi are exact as a pair (TwoProd with fmaf), the cross
//     terms hi*lo + lo*hi are added to the pair's error word, and the pairs
//     are summed with TwoSum (double-float accumulation), across the warp too;
//   * the resulting double-float t is converted to FP64 with integer
//     operations and one FP64 add.
// h_j += a_ij t_i stays a single FP64 FMA per element, so h keeps full FP64
// accumulation.  Power-of-two scalings are exact; h is scaled back by 2^Fz.
// The host takes this kernel only when every column norm is within 2^20 of
// the largest, which keeps every significant entry of A in FP32 range.
// ---------------------------------------------------------------------------

// a * 2^-Eg split into hi + lo (ebias = 896 + Eg).
__device__ __forceinline__ void split_f64(double a, int ebias, float &hi, float &lo) {
  const unsigned hw = (unsigned)__double2hiint(a), lw = (unsigned)__double2loint(a);
  const int ef = (int)((hw >> 20) & 0x7ffu) - ebias;
  const unsigned sign = hw & 0x80000000u;
  const unsigned hib = sign | ((unsigned)ef << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29);
  const int lf = ef - 52;
  const float l = __fmul_rn(__uint2float_rn(lw & 0x1fffffffu), __int_as_float((lf > 0 ? lf : 1) << 23));
  hi = (ef > 0) ? __uint_as_float(hib) : 0.0f;
  lo = (lf > 0) ? __uint_as_float(__float_as_uint(l) | sign) : 0.0f;
}

template <int NC, bool VEC>
__global__ void __launch_bounds__(kPassThreads, NC >= 16 ? 1 : kPassCtasPerSm)
    atax_eft_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int n,
                    const double *__restrict__ z, int ebias, double zscale,
                    double *__restrict__ part, int npad, const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  __shared__ double sh[NC * 64];
  __shared__ double wmax[kPassThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(m, (int64_t)blockIdx.x * per), r1 = min(m, r0 + per);
  // z' = z * 2^Eg, then a common power of two 2^-Fz keeps z'' <= 1.
  double zr[2 * NC];
  load_vec<NC>(z, n, lane, zr);
  double zmax = 0.0;
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) {
    zr[k] *= zscale;
    zmax = fmax(zmax, fabs(zr[k]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) zmax = fmax(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
  if (lane == 0) wmax[warp] = zmax;
  __syncthreads();
  zmax = 0.0;
  for (int w = 0; w < nw; w++) zmax = fmax(zmax, wmax[w]);
  int fz = 0;
  if (zmax > 0.0) frexp(zmax, &fz);
  const double down = ldexp(1.0, -fz), up = ldexp(1.0, fz);
  float zh[2 * NC], zl[2 * NC];
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) {
    const double v = zr[k] * down;
    zh[k] = __double2float_rn(v);
    zl[k] = __double2float_rn(v - (double)zh[k]);
  }
  double h[2 * NC];
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) h[k] = 0.0;
  for (int64_t i = r0 + warp; i < r1; i += nw) {
    double a[2 * NC];
    load_row<NC, VEC>(A + i * lda, n, lane, a);
    float sh_ = 0.0f, sl_ = 0.0f;
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) {
      float ah, al;
      split_f64(a[k], ebias, ah, al);
      const float p = __fmul_rn(ah, zh[k]);
      const float e = __fmaf_rn(ah, zh[k], -p);
      const float c = __fmaf_rn(ah, zl[k], __fmaf_rn(al, zh[k], e));
      float s, err;
      two_sum_f(sh_, p, s, err);
      sh_ = s;
      sl_ = __fadd_rn(sl_, __fadd_rn(err, c));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, sh_, o);
      const float ol = __shfl_xor_sync(0xffffffffu, sl_, o);
      float s, err;
      two_sum_f(sh_, oh, s, err);
      sh_ = s;
      sl_ = __fadd_rn(__fadd_rn(sl_, ol), err);
    }
    const double t = widen(sh_) + widen(sl_);
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) h[k] = fma(a[k], t, h[k]);
  }
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) h[k] *= up;
  cta_store_partial<NC>(h, sh, part, npad);
}

// The FP64 residual pass (lsq_resid.cuh).  With Ahi != NULL it also writes the
// hi / lo FP32 planes of A (the large-problem sketch leaves them to the first
// residual pass of a solve).  Two CTAs per SM up to 8 pairs per lane, one above.
template <int G, int P, bool VEC>
__global__ void __launch_bounds__(kPassThreads, P > 8 ? 1 : kPassCtasPerSm)
    resid_kernel(const ResidArgs a, int64_t m, int n, const double *__restrict__ x,
                 double *__restrict__ part, double *__restrict__ r2_part, int npad,
                 const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  extern __shared__ __align__(16) double rsm[];
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(m, (int64_t)blockIdx.x * per), r1 = min(m, r0 + per);
  resid_body<G, P, VEC>(a, r0, r1, n, x, part + (size_t)blockIdx.x * npad, r2_part + blockIdx.x,
                        npad, rsm);
}

template <int G, int P>
cudaError_t resid_launch(const ResidArgs &a, bool vec, int64_t m, int n, const double *x,
                         double *part, double *r2_part, int grid, int npad, const DevState *gate,
                         cudaStream_t s) {
  constexpr int smem = resid_smem(G, P) * (int)sizeof(double);
  auto *k = vec ? resid_kernel<G, P, true> : resid_kernel<G, P, false>;
  if (smem > 47 * 1024) {  // 48 KB with the static part
    cudaError_t e = ensure_smem_attr((const void *)k, smem);
    if (e != cudaSuccess) return e;
  }
  k<<<grid, kPassThreads, smem, s>>>(a, m, n, x, part, r2_part, npad, gate);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Compensated residual pass (the sketched Karlson-Walden test of Alg. 4's
// second refinement step): r = b - A x and g = A^T r with the compensated dot
// product Dot2 of Ogita, Rump and Oishi (TwoProd by fma, TwoSum, the error
// terms summed alongside), so r and g carry errors of order u |r| and
// u |A^T| |r| rather than the u |A| |x| of a plain FP64 residual, which sits
// at the u ||A||_F threshold of the test.  Per row the lanes' (sum, error)
// pairs are combined with TwoSum across the warp; r = r_hi + r_lo.  Per
// column each lane keeps a (sum, error) pair over its rows; the CTA writes
// both (part2: [grid][2][npad], sums then errors) and reduce_dot2 adds them
// with TwoSum in a fixed order.  About ten FP64 operations per element and
// product, against one.  With cs non-NULL the matrix is fl(A diag(cs)) (the
// column-scaled problem, formed element by element) and x is in its
// coordinates: Alg. 4 runs its test on the scaled problem, where the scaled
// iterate is exact rather than rounded by the change of coordinates.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum_d(double a, double b, double &s, double &e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

template <int NC, bool VEC>
__global__ void __launch_bounds__(kPassThreads, NC >= 8 ? 1 : kPassCtasPerSm)
    resid_dot2_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int n,
                      const double *__restrict__ b, const double *__restrict__ x,
                      const double *__restrict__ cs, double *__restrict__ part2,
                      double *__restrict__ r2_part, int npad) {
  __shared__ double sh[NC * 64];
  __shared__ double csh[NC * 64];
  __shared__ double r2sh[kPassThreads / 32];
  for (int i = threadIdx.x; i < NC * 64; i += blockDim.x) csh[i] = (cs && i < n) ? cs[i] : 1.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(m, (int64_t)blockIdx.x * per), r1 = min(m, r0 + per);
  double xr[2 * NC], gs[2 * NC], gc[2 * NC];
  load_vec<NC>(x, n, lane, xr);
#pragma unroll
  for (int k = 0; k < 2 * NC; k++) gs[k] = gc[k] = 0.0;
  double r2 = 0.0;
  for (int64_t i = r0 + warp; i < r1; i += nw) {
    double a[2 * NC];
    load_row<NC, VEC>(A + i * lda, n, lane, a);
    if (cs) {
#pragma unroll
      for (int k = 0; k < 2 * NC; k++) a[k] *= csh[64 * (k >> 1) + 2 * lane + (k & 1)];
    }
    // this lane's part of b_i - a_i . x (b_i on lane 0)
    double s = (lane == 0) ? b[i] : 0.0, c = 0.0;
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) {
      const double p = -a[k] * xr[k];
      const double ep = fma(-a[k], xr[k], -p);
      double t, es;
      two_sum_d(s, p, t, es);
      s = t;
      c += ep + es;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double os = __shfl_xor_sync(0xffffffffu, s, o);
      const double oc = __shfl_xor_sync(0xffffffffu, c, o);
      double t, es;
      two_sum_d(s, os, t, es);
      s = t;
      c += oc + es;
    }
    double rh, rl;
    two_sum_d(s, c, rh, rl);
    r2 = fma(rh, rh, r2);
#pragma unroll
    for (int k = 0; k < 2 * NC; k++) {
      const double p = a[k] * rh;
      const double ep = fma(a[k], rh, -p);
      double t, es;
      two_sum_d(gs[k], p, t, es);
      gs[k] = t;
      gc[k] += ep + es + a[k] * rl;
    }
  }
  if (lane == 0) r2sh[warp] = r2;
  // the CTA's (sum, error) pairs: sums by TwoSum over the warps in order
  double *ps = part2 + (size_t)blockIdx.x * 2 * npad, *pc = ps + npad;
  for (int i = threadIdx.x; i < NC * 64; i += blockDim.x) sh[i] = 0.0;
  __shared__ double shc[NC * 64];
  for (int i = threadIdx.x; i < NC * 64; i += blockDim.x) shc[i] = 0.0;
  for (int w = 0; w < nw; w++) {
    __syncthreads();
    if (warp == w) {
#pragma unroll
      for (int k = 0; k < 2 * NC; k++) {
        const int col = 64 * (k >> 1) + 2 * lane + (k & 1);
        double t, es;
        two_sum_d(sh[col], gs[k], t, es);
        sh[col] = t;
        shc[col] += gc[k] + es;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < npad; i += blockDim.x) {
    ps[i] = sh[i];
    pc[i] = shc[i];
  }
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < nw; w++) t += r2sh[w];
    r2_part[blockIdx.x] = t;
  }
}

// out[j] = scale[j] (sum_g ps[g][j] + sum_g pc[g][j]) with the sums of the
// partials' sums by TwoSum (one thread per column, a fixed order); *r2 = the
// residual partials' sum.
__global__ void reduce_dot2_kernel(const double *__restrict__ part2, int grid, int npad, int n,
                                   const double *__restrict__ scale, double *__restrict__ out,
                                   const double *__restrict__ r2_part, double *r2) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) {
    double s = 0.0, c = 0.0;
    for (int g = 0; g < grid; g++) {
      double t, es;
      two_sum_d(s, part2[(size_t)g * 2 * npad + j], t, es);
      s = t;
      c += part2[(size_t)g * 2 * npad + npad + j] + es;
    }
    out[j] = scale ? scale[j] * (s + c) : s + c;
  }
  if (r2 != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
    double t = 0.0;
    for (int g = 0; g < grid; g++) t += r2_part[g];
    *r2 = t;
  }
}

// out[c n + j] = scale[j] sum_g part[(c grid + g) npad + j] for c < batch
// (the partials of a batched pass, one block of grid x npad per vector).
__global__ void reduce_batched_kernel(const double *__restrict__ part, int grid, int npad, int n,
                                      int batch, const double *__restrict__ scale,
                                      double *__restrict__ out, const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n * batch) return;
  const int c = (int)(idx / n), j = (int)(idx % n);
  const double *pc = part + (size_t)c * grid * npad + j;
  double s = 0.0;
  for (int g = 0; g < grid; g++) s += pc[(size_t)g * npad];
  out[idx] = scale ? scale[j] * s : s;
}

// out[j] = scale[j] sum_g part[g npad + j]; *r2 = sum_g r2_part[g] (one CTA
// more).  One CTA per 8 columns, 32 threads per column, each the partials
// g = t, t + 32, ...; the 32 sums by shuffles and, across the warps, in
// shared memory (a fixed order, so the result is deterministic).  It is bound
// by latency: a sub-partition issues one FP64 warp instruction per 64 cycles,
// so the n G additions are spread over all SMs.  At G = 304, n = 500: 63 CTAs
// of about 10 additions per thread; CTAs of 32 columns with 38 per thread
// took 6.5 us in the inner loop.
// The partials are written while this kernel waits to start (griddep_wait), so
// they are not __restrict__: the read-only path is for data that no running
// kernel writes.
__global__ void __launch_bounds__(kReduceThreads)
    reduce_kernel(const double *part, int grid, int npad, int n,
                  const double *__restrict__ scale, double *__restrict__ out,
                  const double *r2_part, double *r2, DevState *gate) {
  griddep_launch();
  griddep_wait();
  if (gate != nullptr) {
    const int done = *(volatile const int *)&gate->done;
    if (blockIdx.x == 0 && threadIdx.x == 0) gate->ugate = done;
    if (done) return;
  }
  constexpr int kW = kReduceThreads / 32;
  __shared__ double red[kW][kReduceCols];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (r2 != nullptr && blockIdx.x == gridDim.x - 1) {
    double t = 0.0;
    for (int g = threadIdx.x; g < grid; g += kReduceThreads) t += r2_part[g];
    t = warp_sum(t);
    if (lane == 0) red[warp][0] = t;
    __syncthreads();
    if (warp == 0) {
      t = warp_sum(lane < kW ? red[lane][0] : 0.0);
      if (lane == 0) *r2 = t;
    }
    return;
  }
  const int j0 = blockIdx.x * kReduceCols;
  const double t = sum_partials(part, grid, npad, j0, red);
  if (threadIdx.x < kReduceCols && j0 + threadIdx.x < n)
    out[j0 + threadIdx.x] = scale ? scale[j0 + threadIdx.x] * t : t;
}

bool vec_ok(const double *A, int64_t lda) {
  return ((reinterpret_cast<uintptr_t>(A) & 15) == 0) && (lda % 2 == 0);
}

}  // namespace

#define LSQ_PASS_SWITCH(NPAD, ...)             \
  switch ((NPAD) / 64) {                       \
    case 1: { constexpr int NC = 1; __VA_ARGS__; break; }   \
    case 2: { constexpr int NC = 2; __VA_ARGS__; break; }   \
    case 4: { constexpr int NC = 4; __VA_ARGS__; break; }   \
    case 8: { constexpr int NC = 8; __VA_ARGS__; break; }   \
    case 16: { constexpr int NC = 16; __VA_ARGS__; break; } \
    default: return cudaErrorInvalidValue;     \
  }

cudaError_t launch_pass_atax(const double *A, int64_t lda, int64_t m, int n, const double *z,
                             double *part, int grid, int npad, const DevState *gate,
                             cudaStream_t s) {
  const bool vec = vec_ok(A, lda);
  LSQ_PASS_SWITCH(npad, {
    if (vec) atax_kernel<NC, true><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, z, part, npad, gate);
    else atax_kernel<NC, false><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, z, part, npad, gate);
  });
  return cudaGetLastError();
}

cudaError_t launch_pass_atax_eft(const double *A, int64_t lda, int64_t m, int n, const double *z,
                                 int col_exp, double *part, int grid, int npad,
                                 const DevState *gate, cudaStream_t s) {
  const bool vec = vec_ok(A, lda);
  const int ebias = 896 + col_exp;
  const double zscale = ldexp(1.0, col_exp);
  LSQ_PASS_SWITCH(npad, {
    if (vec) atax_eft_kernel<NC, true><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, z, ebias, zscale, part, npad, gate);
    else atax_eft_kernel<NC, false><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, z, ebias, zscale, part, npad, gate);
  });
  return cudaGetLastError();
}

cudaError_t launch_pass_resid(const double *A, int64_t lda, int64_t m, int n, const double *b,
                              const double *x, double *part, double *r2_part, int grid, int npad,
                              cudaStream_t s, float *Ahi, float *Alo, int64_t ld32,
                              const DevState *gate, const double *bscale, double *rout) {
  const bool vec = vec_ok(A, lda);
  const ResidArgs a = {A, lda, b, bscale, rout, Ahi, Alo, ld32};
  const DfTile t = df_tile(n);
  switch (t.G * 100 + t.P) {
#define LSQ_RES(GV, PV) \
  case GV * 100 + PV:   \
    return resid_launch<GV, PV>(a, vec, m, n, x, part, r2_part, grid, npad, gate, s);
    LSQ_RES(8, 1) LSQ_RES(8, 2) LSQ_RES(8, 3) LSQ_RES(8, 4) LSQ_RES(8, 5) LSQ_RES(8, 6)
    LSQ_RES(8, 7) LSQ_RES(8, 8) LSQ_RES(16, 5) LSQ_RES(16, 6) LSQ_RES(16, 7) LSQ_RES(16, 8)
    LSQ_RES(32, 5) LSQ_RES(32, 6) LSQ_RES(32, 7) LSQ_RES(32, 8) LSQ_RES(32, 10) LSQ_RES(32, 12)
    LSQ_RES(32, 14) LSQ_RES(32, 16)
#undef LSQ_RES
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_pass_resid_dot2(const double *A, int64_t lda, int64_t m, int n,
                                   const double *b, const double *x, const double *cs,
                                   double *part2, double *r2_part, int grid, int npad,
                                   cudaStream_t s) {
  const bool vec = vec_ok(A, lda);
  LSQ_PASS_SWITCH(npad, {
    if (vec)
      resid_dot2_kernel<NC, true><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, b, x, cs, part2,
                                                                r2_part, npad);
    else
      resid_dot2_kernel<NC, false><<<grid, kPassThreads, 0, s>>>(A, lda, m, n, b, x, cs, part2,
                                                                 r2_part, npad);
  });
  return cudaGetLastError();
}

cudaError_t launch_reduce_dot2(const double *part2, int grid, int npad, int n, const double *scale,
                               double *out, const double *r2_part, double *r2, cudaStream_t s) {
  reduce_dot2_kernel<<<(n + 127) / 128, 128, 0, s>>>(part2, grid, npad, n, scale, out, r2_part, r2);
  return cudaGetLastError();
}

cudaError_t launch_reduce_batched(const double *part, int grid, int npad, int n, int batch,
                                  const double *scale, double *out, const DevState *gate,
                                  cudaStream_t s) {
  const int64_t cnt = (int64_t)n * batch;
  reduce_batched_kernel<<<(unsigned)((cnt + 127) / 128), 128, 0, s>>>(part, grid, npad, n, batch,
                                                                      scale, out, gate);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const double *part, int grid, int npad, int n, const double *scale,
                          double *out, const double *r2_part, double *r2, DevState *gate,
                          cudaStream_t s) {
  const int g = (n + kReduceCols - 1) / kReduceCols + (r2 != nullptr ? 1 : 0);
  if (gate != nullptr)
    return launch_pdl(reduce_kernel, dim3(g), dim3(kReduceThreads), 0, s, part, grid, npad, n,
                      scale, out, r2_part, r2, gate);
  reduce_kernel<<<g, kReduceThreads, 0, s>>>(part, grid, npad, n, scale, out, r2_part, r2, gate);
  return cudaGetLastError();
}

}  // namespace lsq
