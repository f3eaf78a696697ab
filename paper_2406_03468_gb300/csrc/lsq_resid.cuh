// The FP64 residual pass r = b - A x, A^T r, ||r||^2 of one CTA, shared by the
// plans (k_pass.cu) and the batched engine (k_batch.cu).
//
// Bound by the FP64 pipe (a sub-partition issues one FP64 warp instruction per
// 64 cycles): 4 P instructions for the 32 / G rows a warp takes at a time, and
// log2 G + 2 for the row sums' reduction and r.  So, as in the double-float pass
// (lsq_dfpass.cuh), G lanes share a row and hold P pairs of its columns, with
// the smallest G that covers n in 8 pairs: no instruction works on columns
// beyond the next multiple of 2 G, and the reduction is shared by 32 / G rows.
// FP64 instructions per row, one row per warp in tiles of 64, 128, 256, 512 or
// 1024 columns / here: n = 32 11 / 3.3, n = 64 11 / 5.3, n = 128 15 / 9.3, n = 333
// 39 / 31, n = 500 39 / 39.  The same reads of A also give the FP32 planes
// (Ahi != NULL): HBM has room under this pass.
#pragma once
#include "lsq_dfpass.cuh"

namespace lsq {

// doubles of shared memory: one FP64 sum per warp and column
constexpr int resid_smem(int G, int P) { return kDfWarps * 2 * G * P; }

struct ResidArgs {
  const double *A;
  int64_t lda;
  const double *b;
  const double *bscale;  // NULL: 1
  double *rout;          // NULL: r is not kept (may be b)
  float *Ahi, *Alo;
  int64_t ld32;
};

template <int G, int P, bool VEC>
__device__ __forceinline__ void resid_body(const ResidArgs &a, int64_t r0, int64_t r1, int n,
                                           const double *__restrict__ x, double *part,
                                           double *r2_out, int npad, double *sh) {
  constexpr int RPW = 32 / G, kCols = 2 * G * P;
  __shared__ double r2sh[kDfWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = lane % G, grp = lane / G;
  const double bs = a.bscale != nullptr ? *a.bscale : 1.0;
  double xr[2 * P], g[2 * P];
#pragma unroll
  for (int k = 0; k < P; k++) {
    const int col = 2 * G * k + 2 * gl;
    xr[2 * k] = col < n ? x[col] : 0.0;
    xr[2 * k + 1] = col + 1 < n ? x[col + 1] : 0.0;
    g[2 * k] = g[2 * k + 1] = 0.0;
  }
  double r2 = 0.0;
  for (int64_t i0 = r0 + RPW * warp; i0 < r1; i0 += RPW * kDfWarps) {
    const int64_t i = i0 + grp;
    const bool ok = i < r1;
    const double *row = a.A + (ok ? i : i0) * a.lda;
    double v[2 * P];
#pragma unroll
    for (int k = 0; k < P; k++) {
      const int col = 2 * G * k + 2 * gl;
      if (VEC && col + 1 < n) {
        const double2 w = __ldcs(reinterpret_cast<const double2 *>(row + col));
        v[2 * k] = w.x;
        v[2 * k + 1] = w.y;
      } else {
        v[2 * k] = col < n ? __ldcs(row + col) : 0.0;
        v[2 * k + 1] = col + 1 < n ? __ldcs(row + col + 1) : 0.0;
      }
    }
    const double bi = ok ? a.b[i] : 0.0;
    if (a.Ahi != nullptr && ok) {
#pragma unroll
      for (int k = 0; k < P; k++) {
        const int col = 2 * G * k + 2 * gl;
        float h0, l0, h1, l1;
        split_rn(v[2 * k], h0, l0);
        split_rn(v[2 * k + 1], h1, l1);
        if (col + 1 < n) {
          __stcs(reinterpret_cast<float2 *>(a.Ahi + i * a.ld32 + col), make_float2(h0, h1));
          __stcs(reinterpret_cast<float2 *>(a.Alo + i * a.ld32 + col), make_float2(l0, l1));
        } else if (col < n) {
          __stcs(a.Ahi + i * a.ld32 + col, h0);
          __stcs(a.Alo + i * a.ld32 + col, l0);
        }
      }
    }
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < P; k++) {
      s0 = fma(v[2 * k], xr[2 * k], s0);
      s1 = fma(v[2 * k + 1], xr[2 * k + 1], s1);
    }
    double s = s0 + s1;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double r = ok ? (a.bscale != nullptr ? bs * bi : bi) - s : 0.0;
    if (a.rout != nullptr) {
      __syncwarp();  // every lane has read b (rout may be b)
      if (ok && gl == 0) a.rout[i] = r;
    }
    r2 = fma(r, r, r2);
#pragma unroll
    for (int k = 0; k < 2 * P; k++) g[k] = fma(v[k], r, g[k]);
  }
  // the groups' column sums added to each other, halving the pairs a lane
  // holds (lanes 16 apart, then 8), then the warp's sums to shared memory and
  // the CTA's in warp order
  constexpr int PA = RPW > 1 ? (P + 1) / 2 : P, PB = RPW > 2 ? (PA + 1) / 2 : PA;
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  if (RPW > 1) {
#pragma unroll
    for (int k = 0; k < PA; k++)
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const double even = g[4 * k + e], odd = 2 * k + 1 < P ? g[2 * k + 1 < P ? 4 * k + 2 + e : 0] : 0.0;
        g[2 * k + e] = (h16 ? odd : even) + __shfl_xor_sync(0xffffffffu, h16 ? even : odd, 16);
      }
  }
  if (RPW > 2) {
#pragma unroll
    for (int k = 0; k < PB; k++)
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const double even = g[4 * k + e], odd = 2 * k + 1 < PA ? g[2 * k + 1 < PA ? 4 * k + 2 + e : 0] : 0.0;
        g[2 * k + e] = (h8 ? odd : even) + __shfl_xor_sync(0xffffffffu, h8 ? even : odd, 8);
      }
  }
#pragma unroll
  for (int k = 0; k < PB; k++) {
    int pk = k;
    if (RPW > 2) pk = 2 * pk + (h8 ? 1 : 0);
    if (RPW > 1) pk = 2 * pk + (h16 ? 1 : 0);
    if (pk < P) {
      sh[warp * kCols + 2 * G * pk + 2 * gl] = g[2 * k];
      sh[warp * kCols + 2 * G * pk + 2 * gl + 1] = g[2 * k + 1];
    }
  }
  r2 = warp_sum(gl == 0 ? r2 : 0.0);
  if (lane == 0) r2sh[warp] = r2;
  __syncthreads();
  for (int c = threadIdx.x; c < kCols && c < npad; c += kPassThreads) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kDfWarps; w++) t += sh[w * kCols + c];
    part[c] = t;
  }
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kDfWarps; w++) t += r2sh[w];
    *r2_out = t;
  }
}

}  // namespace lsq
