// The inner passes over the FP32 planes of A for one problem (lsq_dfpass.cuh
// holds their body): atax_df (double-float), atax32 (the FP32 tier) and LSQR's
// pass.  A CTA takes a contiguous range of rows and writes its partial sums;
// reduce_kernel (k_pass.cu) adds them in a fixed order.
#include <algorithm>

#include "lsq_dfpass.cuh"

namespace lsq {

namespace {

struct DfArgs {
  const float *Ahi, *Alo;
  int ld32;
  int64_t m;
  int n;
  const double *z;
  double *s;
  const double *bscale;
  double *part, *r2part;
  int npad;
  const DevState *gate;
  int *err;
  bool keep;
  int64_t zstride, pstride;
};

// Two CTAs per SM up to 8 pairs per lane (128 registers), one above.
template <int G, int P, int MODE>
__global__ void __launch_bounds__(kPassThreads, P > 8 ? 1 : kPassCtasPerSm)
    df_pass_kernel(const DfArgs a) {
  griddep_launch();
  extern __shared__ __align__(16) double dsm[];
  const int64_t per = (a.m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(a.m, (int64_t)blockIdx.x * per), r1 = min(a.m, r0 + per);
  // many right-hand sides: grid row blockIdx.y works on vector z_(blockIdx.y)
  df_pass_body<G, P, MODE>(a.Ahi, a.Alo, a.ld32, r0, r1, a.n, a.z + blockIdx.y * a.zstride, a.s,
                           a.bscale,
                           a.part + blockIdx.y * a.pstride + (size_t)blockIdx.x * a.npad,
                           a.r2part + blockIdx.x, a.npad,
                           a.gate != nullptr ? &a.gate->done : nullptr, a.err, a.keep, dsm);
}

template <int G, int P, int MODE>
cudaError_t df_launch(const DfArgs &a, dim3 grid, cudaStream_t s) {
  constexpr size_t smem = df_smem(G, P, MODE);
  auto *k = df_pass_kernel<G, P, MODE>;
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem_attr((const void *)k, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (a.gate != nullptr) return launch_pdl(k, grid, dim3(kPassThreads), smem, s, a);
  k<<<grid, kPassThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t df_dispatch(const DfArgs &a, dim3 grid, cudaStream_t s) {
  const DfTile t = df_tile(a.n);
  switch (t.G * 100 + t.P) {
#define LSQ_DF(GV, PV) \
  case GV * 100 + PV:  \
    return df_launch<GV, PV, MODE>(a, grid, s);
    LSQ_DF(8, 1) LSQ_DF(8, 2) LSQ_DF(8, 3) LSQ_DF(8, 4) LSQ_DF(8, 5) LSQ_DF(8, 6) LSQ_DF(8, 7)
    LSQ_DF(8, 8) LSQ_DF(16, 5) LSQ_DF(16, 6) LSQ_DF(16, 7) LSQ_DF(16, 8) LSQ_DF(32, 5)
    LSQ_DF(32, 6) LSQ_DF(32, 7) LSQ_DF(32, 8) LSQ_DF(32, 10) LSQ_DF(32, 12) LSQ_DF(32, 14)
    LSQ_DF(32, 16)
#undef LSQ_DF
    default:
      return cudaErrorInvalidValue;
  }
}

bool df_keep(int64_t m, int64_t ld32, int planes) {
  return (double)m * (double)ld32 * 4.0 * planes <= kL2KeepBytes;
}

}  // namespace

// grid: two CTAs per SM.  Above n = 512 one is resident, so a second wave would
// only repeat the prologue and the flush.  Short problems take fewer CTAs: a
// CTA's fixed costs (z's split, the last flush) and the reduction's partial
// sums weigh more than its rows, and the waiting small kernels find room on
// the SMs.  us per iteration at 3/8, 3/4 and 1 of the grid: 20000 x 97 16.8,
// 17.3, 21.9; 60000 x 97 27.4, 25.6, 28.6; 120000 x 128 (1/2, 3/4, 1) 55.1,
// 42.5, 38.5; 8000 x 500 (1/2, 1) 25.5, 31.6; 32000 x 500 56.0, 44.5.
int pass_df_grid(int64_t m, int n, int64_t ld32, int grid) {
  const DfTile t = df_tile(n);
  const int64_t blocks = (m + df_block_rows(t, (int)ld32) - 1) / df_block_rows(t, (int)ld32);
  const double per_warp = (double)blocks / ((double)grid * kDfWarps);
  int g = grid;
  if (t.P > 8) g = grid / 2;
  else if (t.G == 32) g = per_warp < 8.0 ? grid / 2 : grid;
  else g = per_warp < 2.5 ? 3 * grid / 8 : per_warp < 10.0 ? 3 * grid / 4 : grid;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, (blocks + kDfWarps - 1) / kDfWarps));
}

cudaError_t launch_pass_atax_df(const float *Ahi, const float *Alo, int64_t ld32, int64_t m, int n,
                                const double *z, double *part, int grid, int npad,
                                const DevState *gate, int *err, cudaStream_t s, int batch,
                                int64_t zstride, int64_t pstride) {
  const DfArgs a = {Ahi, Alo, (int)ld32, m, n, z, nullptr, nullptr, part, nullptr, npad, gate, err,
                    df_keep(m, ld32, 2), zstride, pstride};
  return df_dispatch<0>(a, dim3(grid, batch), s);
}

cudaError_t launch_pass_lsqr_df(const float *Ahi, const float *Alo, int64_t ld32, int64_t m, int n,
                                const double *z, double *sv, const double *bscale, double *part,
                                double *r2part, int grid, int npad, const DevState *gate, int *err,
                                cudaStream_t s) {
  const DfArgs a = {Ahi, Alo, (int)ld32, m, n, z, sv, bscale, part, r2part, npad, gate, err,
                    df_keep(m, ld32, 2), 0, 0};
  return df_dispatch<1>(a, dim3(grid), s);
}

cudaError_t launch_pass_atax32(const float *A32, int64_t ld32, int64_t m, int n, const double *z,
                               double *part, int grid, int npad, const DevState *gate, int *err,
                               cudaStream_t s) {
  const DfArgs a = {A32, nullptr, (int)ld32, m, n, z, nullptr, nullptr, part, nullptr, npad, gate,
                    err, df_keep(m, ld32, 1), 0, 0};
  return df_dispatch<2>(a, dim3(grid), s);
}

}  // namespace lsq
