// Streaming passes of a batch of problems solved in lockstep (lsq_batch.cu):
// one launch covers every item, CTA g working on rows of item cta_item[g]
// (the CTAs are dealt to the items in proportion to their m n).  Per item the
// arithmetic is the single-problem passes' (k_pass.cu):
//   b_resid:  r = b - A x, partial sums of A^T r and ||r||^2, all FP64;
//   b_inner:  partial sums of A^T (A z) in double-float on the item's hi / lo
//             FP32 planes (TwoProd / TwoSum on packed f32x2 pairs, the column
//             sums flushed into FP64 every 32 rows), z scaled by a power of two;
//   b_reduce: the item's partials summed in a fixed order, times D^-1.
// n <= 256 (npad 64, 128 or 256).  The inner pass returns at once for an
// item whose inner loop has stopped (st->done), so the launch costs nothing
// for the items that are done.
#include "lsq_common.cuh"
#include "lsq_resid.cuh"

namespace lsq {

namespace {

constexpr int kBThreads = kPassThreads;

// The FP64 residual pass of one item's CTA (lsq_resid.cuh).  The planes are
// the sketch's.
__global__ void __launch_bounds__(kBThreads, 2)
    b_resid_kernel(const BItem *__restrict__ items, const int *__restrict__ cta_item) {
  __shared__ double sh[resid_smem(16, 8)];
  const int idx = cta_item[blockIdx.x];
  if (idx < 0) return;
  const BItem &it = items[idx];
  const int local = blockIdx.x - it.cta0;
  const int64_t per = (it.m + it.ncta - 1) / it.ncta;
  const int64_t r0 = min(it.m, (int64_t)local * per), r1 = min(it.m, r0 + per);
  const ResidArgs a = {it.A, it.n, it.b, nullptr, nullptr, nullptr, nullptr, 0};
  const bool vec = (reinterpret_cast<uintptr_t>(it.A) & 15) == 0 && it.n % 2 == 0;
  double *part = it.part + (size_t)local * it.npad, *r2 = it.r2part + local;
  const DfTile t = df_tile(it.n);
  switch (t.G * 100 + t.P) {
#define LSQ_BRES(GV, PV)                                                                \
  case GV * 100 + PV:                                                                   \
    if (vec) resid_body<GV, PV, true>(a, r0, r1, it.n, it.xo, part, r2, it.npad, sh);   \
    else resid_body<GV, PV, false>(a, r0, r1, it.n, it.xo, part, r2, it.npad, sh);      \
    break;
    LSQ_BRES(8, 1) LSQ_BRES(8, 2) LSQ_BRES(8, 3) LSQ_BRES(8, 4) LSQ_BRES(8, 5) LSQ_BRES(8, 6)
    LSQ_BRES(8, 7) LSQ_BRES(8, 8) LSQ_BRES(16, 5) LSQ_BRES(16, 6) LSQ_BRES(16, 7) LSQ_BRES(16, 8)
#undef LSQ_BRES
    default: break;
  }
}

// The inner pass of one item's CTA over the item's row share (lsq_dfpass.cuh),
// in the tile its n takes (at most 8 pairs of columns per lane: n <= 256).
__global__ void __launch_bounds__(kBThreads, 2)
    b_inner_kernel(const BItem *__restrict__ items, const int *__restrict__ cta_item) {
  extern __shared__ __align__(16) double dsm[];
  const int idx = cta_item[blockIdx.x];
  if (idx < 0) return;
  const BItem &it = items[idx];
  if (*(volatile const int *)&it.st->done) return;
  const int local = blockIdx.x - it.cta0;
  const int64_t per = (it.m + it.ncta - 1) / it.ncta;
  const int64_t r0 = min(it.m, (int64_t)local * per), r1 = min(it.m, r0 + per);
  const DfTile t = df_tile(it.n);
  switch (t.G * 100 + t.P) {
#define LSQ_BDF(GV, PV)                                                                         \
  case GV * 100 + PV:                                                                           \
    df_pass_body<GV, PV, 0>(it.Ahi, it.Alo, it.ld32, r0, r1, it.n, it.z, nullptr, nullptr,      \
                            it.part + (size_t)local * it.npad, nullptr, it.npad, nullptr,       \
                            &it.st->err, false, dsm);                                           \
    break;
    LSQ_BDF(8, 1) LSQ_BDF(8, 2) LSQ_BDF(8, 3) LSQ_BDF(8, 4) LSQ_BDF(8, 5) LSQ_BDF(8, 6)
    LSQ_BDF(8, 7) LSQ_BDF(8, 8) LSQ_BDF(16, 5) LSQ_BDF(16, 6) LSQ_BDF(16, 7) LSQ_BDF(16, 8)
#undef LSQ_BDF
    default: break;
  }
}

// out[j] = dinv[j] sum_g part[g npad + j] over the item's CTAs (8 warps per
// 32 columns, each summing every 8th partial, then one warp adds the 8 in
// order); mode 0 also *r2 = sum of the residual partials.  Grid (column
// blocks, items).
__global__ void __launch_bounds__(256)
    b_reduce_kernel(const BItem *__restrict__ items, int mode) {
  __shared__ double red[8][33];
  const BItem &it = items[blockIdx.y];
  if (mode == 1) {
    const int done = *(volatile const int *)&it.st->done;
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // for the kernels behind (k_inner.cu)
      it.st->ugate = done;
      it.st->par = it.st->iters & 1;
    }
    if (done) return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  if (blockIdx.x * 32 >= it.n && !(mode == 0 && blockIdx.x == 0)) return;
  double s = 0.0;
  if (j < it.n)
    for (int g = warp; g < it.ncta; g += 8) s += it.part[(size_t)g * it.npad + j];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && j < it.n) {
    double t = 0.0;
    for (int w = 0; w < 8; w++) t += red[w][lane];
    (mode == 0 ? it.g : it.h)[j] = it.dinv[j] * t;
  }
  if (mode == 0 && blockIdx.x == 0) {
    __syncthreads();
    double t = 0.0;
    for (int g = threadIdx.x; g < it.ncta; g += 256) t += it.r2part[g];
    t = warp_sum(t);
    if (lane == 0) red[warp][32] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double u = 0.0;
      for (int w = 0; w < 8; w++) u += red[w][32];
      it.st->r2 = u;
    }
  }
}

// Deal the `grid` CTAs of the row-parallel passes to the items in proportion
// to m n: every item (all = 1) or only the items whose inner loop is still
// running (all = 0), so that the last items of a batch get the whole GPU.
// Writes cta0 / ncta of the table and the CTA -> item map (-1: no item).
// One CTA of 256 threads, one per item (count <= 256).
__global__ void __launch_bounds__(256)
    b_redeal_kernel(BItem *__restrict__ items, int count, int *__restrict__ cta_item, int grid,
                    int all) {
  __shared__ double scratch[8];
  __shared__ int wcnt[8], woff[8];
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  const bool on = i < count && (all || !*(volatile const int *)&items[i].st->done);
  const double mn = on ? (double)items[i].m * items[i].n : 0.0;
  const double tot = block_sum(mn, scratch);
  // the item's rank among the active ones, and their number
  auto rank = [&](int v, int &total) {  // exclusive prefix sum over the CTA
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) wcnt[warp] = x;
    __syncthreads();
    if (i < 8) {
      int b = 0;
      for (int w = 0; w < i; w++) b += wcnt[w];
      woff[i] = b;
    }
    __syncthreads();
    total = woff[7] + wcnt[7];
    return woff[warp] + x - v;
  };
  int act = 0, used = 0, end = 0;
  const int r = rank(on ? 1 : 0, act);
  int c = on ? 1 : 0;
  if (on && grid > act) c += (int)floor(mn / tot * (grid - act));
  rank(c, used);
  // the rest one at a time, in item order
  if (on && act > 0 && grid > used) c += (grid - used) / act + (r < (grid - used) % act ? 1 : 0);
  const int c0 = rank(c, end);
  if (i < count) {
    items[i].cta0 = c0;
    items[i].ncta = c;
  }
  for (int k = 0; k < c; k++) cta_item[c0 + k] = i;
  for (int k = end + i; k < grid; k += 256) cta_item[k] = -1;
}

// Zero every item's sketch accumulator SAb (d x (n + 1)) before the scatter.
__global__ void b_zero_kernel(const BItem *__restrict__ items) {
  const BItem &it = items[blockIdx.y];
  const int64_t cnt = (int64_t)it.d * (it.n + 1);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x)
    it.SAb[i] = 0.0;
}

}  // namespace

cudaError_t launch_b_redeal(BItem *items, int count, int *cta_item, int grid, int all,
                            cudaStream_t s) {
  if (count > 256) return cudaErrorInvalidValue;
  b_redeal_kernel<<<1, 256, 0, s>>>(items, count, cta_item, grid, all);
  return cudaGetLastError();
}

cudaError_t launch_b_zero(const BItem *items, int count, cudaStream_t s) {
  b_zero_kernel<<<dim3(64, count), 256, 0, s>>>(items);
  return cudaGetLastError();
}

cudaError_t launch_b_resid(const BItem *items, const int *cta_item, int grid, cudaStream_t s) {
  b_resid_kernel<<<grid, kBThreads, 0, s>>>(items, cta_item);
  return cudaGetLastError();
}

cudaError_t prepare_b_inner() {
  return ensure_smem_attr((const void *)b_inner_kernel, (int)df_smem(16, 8, 0));
}

cudaError_t launch_b_inner(const BItem *items, const int *cta_item, int grid, cudaStream_t s) {
  b_inner_kernel<<<grid, kBThreads, df_smem(16, 8, 0), s>>>(items, cta_item);
  return cudaGetLastError();
}

cudaError_t launch_b_reduce(const BItem *items, int count, int nmax, int mode, cudaStream_t s) {
  b_reduce_kernel<<<dim3((nmax + 31) / 32, count), 256, 0, s>>>(items, mode);
  return cudaGetLastError();
}

}  // namespace lsq
