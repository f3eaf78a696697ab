// Inner pass for many right-hand sides, H = A^T (A Z) for up to 64 vectors, on
// the tensor cores (tcgen05, FP32 accumulators in TMEM) in fixed point.
//
// GB300's FP64 tensor rate is about 1 TFLOP/s and the double-float form on the
// FP32 pipe (k_multi_df.cu) takes 24 packed operations per element and pair of
// vectors: 5.9 ms per pass at 500000 x 200 x 64.  Here every operand is an
// integer of 56 bits written in 7 balanced digits of 8 bits (-128 .. 128), each
// digit exact in bf16:
//   A:  a_ij = q 2^(E_j - g_i - 55), |a_ij| < 2^(E_j - g_i): E_j the column's
//       largest exponent, g_i >= 0 the row's gap below the columns' largest
//       (rows whose entries are all small keep all of their bits: they can be
//       the ones that determine a direction of x);
//   z:  v_jc = 2^E_j z_jc = q 2^(F_c - 55), |v_jc| < 2^F_c;
//   y = A z: 2^g_i y_i in units of 2^(F_c - 54), then 2^-g_i y_i per vector against
//       its largest entry (|A| |z| can be kappa times |A z|), A^T y being
//       2^E_j times the sum over i of (2^(g_i - E_j) a_ij) (2^-g_i y_i).
// A product of two integers is the sum over digit pairs (t, s) of weight
// 256^(12 - t - s).  The inner pass keeps the 28 pairs with t + s <= 6: what is
// dropped is 2^-56.3 (rms of random digits; 2^-53.4 at most) of the largest
// product per term, 2^-52.5 over 200 full-scale terms.  The residual pass, which
// stands in for FP64 sums, keeps the 34 with t + s <= 7 (dropped: 2^-61.7 at most):
// with 28 its answers were up to 2.9 times further off than with FP64 residual
// passes (n = 16, kappa 1e3 .. 1e6; 3.8 times with one large entry per row), with
// 34 they are no further off (1e6, consistent: 0.4 times).  The pairs of one weight
// share an accumulator: products are at most 2^14 and the sums at most 2^24 for the
// 4 leading weights over 256 columns or rows, so FP32 accumulation is exact there;
// the others reach 2^24 and round only where the digits of many terms are all
// large and of one sign, at 2^-49 of the result's scale.  The accumulators (7 or 8)
// are combined in 64-bit integers.  An entry's error is 2^-56 of 2^(E_j - g_i),
// against 2^-48 of the entry for the FP32 planes: no larger while a column's
// typical (geometric mean) entry is within 2^8 of that (Gaussian matrices: 2^1.5 ..
// 2^3.1), else the driver takes the double-float form; the residual pass needs 2^5
// (multi_tc_columns_ok).  Per row, A x of the residual pass is off by 2^-54 .. 2^-57
// of |A| |x| (rms; sequential FP64 sums: 2^-53 .. 2^-55; n = 16 .. 200, graded x, one
// large entry per row, rows graded by 2^30).  Measured at kappa = 1e1 .. 1e10:
// backward errors 1e-17; A^T (A z) of the inner pass off by 9e-17 of |A|^T |A z|
// (double-float: 3e-15).
//
// Both products are the same GEMM, D[128 x 64] += P^(t)[128 x K] Q^(s)[64 x K]^T:
//   y:  P = A (rows i, K = columns j),     Q = Z^T  -> y in 64 bits and each
//       vector's largest; tc_yprep_kernel writes y's digits
//   h:  P = A^T (rows j, K = rows i),      Q = Y^T  -> 64-bit partial sums
// A's digits are kept in both layouts, written once per solve, in the tiles
// that the tensor cores read (128 rows of 64 bf16, 128-byte swizzle, 16 KB):
// a tile is one contiguous bulk copy.  A CTA (one per SM) runs a producer warp
// (copies: a ring of P tiles, two sets of Q tiles), an issuing warp (one thread)
// and sixteen warps that read the accumulators (7 or 8 x 64 columns of TMEM).
//
// Measured: see launch_multi_tc_pass.  Every wait is bounded; on a timeout
// the CTA records LSQ_ERR_TIMEOUT, waits (bounded) for its copies and MMAs,
// frees its TMEM and returns.
#include <algorithm>

#include "lsq_common.cuh"
#include "lsq_dev.cuh"

namespace lsq {

namespace {

constexpr int kS = 7;                       // digits
constexpr int kPTile = 128 * 64 * 2;        // bytes of a P tile
constexpr int kPStages = 6;
constexpr int kTcThreads = 576;             // producer, issuer, 16 epilogue warps
constexpr int kTcBad = 1 << 20;
constexpr int kNoGap = 1 << 20;               // a row of zeros
constexpr int kNoBits = -8192;                // below every row's bits of y minus its gaps
// h: 256 rows per accumulation.  The d + 1 digit pairs of weight d add up to
// (d + 1) 2^14 256 <= 2^24 for d <= 3, whatever the digits: exact in FP32.  (1024
// rows take 8% less time per pass, but weights 1 .. 3 round, at 2^-32 .. 2^-48, where
// the digits of many rows are all large and of one sign.)
constexpr int kFlushChunks = 4;
constexpr uint64_t kTcWaitNs = 1000ull * 1000 * 1000;  // 1 s

__host__ __device__ constexpr int tc_qset(int nv) { return kS * nv * 128; }  // bytes, nv vectors

// The first layout's last column chunk, when n leaves it w = 16 ks < 64 columns,
// holds 4 / ks digits side by side in a tile (n = 200: 23 tiles per row tile
// instead of 28).
struct TcCols {
  int nkc;   // chunks of 64 columns
  int ks;    // K steps of 16 in the last one
  int dpt;   // its digits per tile
  int tiles; // tiles of a row tile
};
inline __host__ __device__ TcCols tc_cols(int n) {
  TcCols t;
  t.nkc = (n + 63) / 64;
  t.ks = (n - 64 * (t.nkc - 1) + 15) / 16;
  t.dpt = 4 / t.ks;
  t.tiles = (t.nkc - 1) * kS + (kS + t.dpt - 1) / t.dpt;
  return t;
}

// byte of element (row r, column k) of a tile of rows of 64 bf16
__device__ __forceinline__ unsigned tc_off(int r, int k) {
  return (unsigned)(r * 128 + (((k >> 3) ^ (r & 7)) << 4) + ((k & 7) << 1));
}

// The kS balanced digits of q0 and q1 as bf16, a pair per word.  128 added to
// each of the 6 lower digits makes them bytes; 2^23 + 2^22 + b in FP32 holds b in
// its low byte, and subtracting 2^23 + 2^22 + 128 leaves the digit as a float, of
// which bf16 keeps all bits (exact up to 256).
__device__ __forceinline__ void tc_digits(long long q0, long long q1, unsigned (&w)[kS]) {
  const unsigned long long u0 = (unsigned long long)q0 + 0x808080808080ull;
  const unsigned long long u1 = (unsigned long long)q1 + 0x808080808080ull;
  const unsigned lo0 = (unsigned)u0, hi0 = (unsigned)(u0 >> 32);
  const unsigned lo1 = (unsigned)u1, hi1 = (unsigned)(u1 >> 32);
#pragma unroll
  for (int s = 0; s < kS; s++) {
    const int k = kS - 1 - s;  // byte
    const float f0 =
        s == 0 ? __int_as_float(0x4b400000 + ((int)hi0 >> 16)) - 12582912.0f
               : __uint_as_float(__byte_perm(k < 4 ? lo0 : hi0, 0x4b400000u, 0x7640 | (k & 3))) -
                     12583040.0f;
    const float f1 =
        s == 0 ? __int_as_float(0x4b400000 + ((int)hi1 >> 16)) - 12582912.0f
               : __uint_as_float(__byte_perm(k < 4 ? lo1 : hi1, 0x4b400000u, 0x7640 | (k & 3))) -
                     12583040.0f;
    w[s] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
  }
}

// q 2^-sh rounded to an integer, |q 2^-sh| <= 2^55 (or q = 0).  No branches: the
// rows of a warp differ in sh.
__device__ __forceinline__ long long shift_round(long long q, int sh) {
  const long long r = q >> min(max(sh - 1, 0), 63), l = q << min(max(1 - sh, 0), 63);
  return ((sh > 0 ? r : l) + 1) >> 1;
}

// v 2^-g for g >= 0, zero below the normal range (integer operations: FP64 ones
// take 64 cycles per warp)
__device__ __forceinline__ double scale_down(double v, int g) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7ff);
  return e == 0x7ff ? v : e <= g ? 0.0 : __longlong_as_double(b - ((long long)g << 52));
}

// |a| 2^(55 - E) rounded to an integer, with a's sign (|a| < 2^E)
__device__ __forceinline__ long long tc_fix(double a, int E) {
  const long long b = __double_as_longlong(a);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return 0;
  const long long mant = (b & 0xfffffffffffffll) | 0x10000000000000ll;
  const int sh = ex - 1075 + 55 - E;  // at most 2
  long long q;
  if (sh >= 0) q = mant << min(sh, 8);
  else if (sh > -60) q = (mant + (1ll << (-sh - 1))) >> -sh;
  else q = 0;
  return b < 0 ? -q : q;
}

// Per column: the largest biased exponent.
__global__ void __launch_bounds__(256)
    tc_colmax_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int n, TcCol *col) {
  const int j = threadIdx.x;
  if (j >= n) return;
  int e = 0;
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(m, r0 + per);
#pragma unroll 8
  for (int64_t i = r0; i < r1; i++)
    e = max(e, (__double2hiint(__ldcs(A + i * lda + j)) >> 20) & 0x7ff);
  atomicMax(&col[j].emax, e);
}

// Per row its gap g_i, the powers of two that its entry nearest to its column's
// largest lies below it (0 for a row of zeros and beyond m); and per column the
// number of entries that are not zero and the sum of the powers of two that they
// lie below 2^(E_j - g_i).  A warp per row; bound by the read of A.
__global__ void __launch_bounds__(256)
    tc_rowgap_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int64_t mp, int n,
                     TcCol *col, short *__restrict__ gap) {
  __shared__ unsigned long long sums[256];
  __shared__ int cnts[256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  sums[threadIdx.x] = 0;
  cnts[threadIdx.x] = 0;
  int em[8], cnt[8];
  long long sum[8];
#pragma unroll
  for (int k = 0; k < 8; k++) {
    em[k] = 32 * k + lane < n ? col[32 * k + lane].emax : 0;
    cnt[k] = 0;
    sum[k] = 0;
  }
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * 8 + warp; i < mp; i += (int64_t)gridDim.x * 8) {
    int x[8], g = kNoGap;
#pragma unroll
    for (int k = 0; k < 8; k++)
      x[k] = i < m && 32 * k + lane < n
                 ? (__double2hiint(__ldcs(A + i * lda + 32 * k + lane)) >> 20) & 0x7ff : 0;
#pragma unroll
    for (int k = 0; k < 8; k++)
      if (x[k] != 0) g = min(g, em[k] - x[k]);
    g = __reduce_min_sync(0xffffffffu, g);
#pragma unroll
    for (int k = 0; k < 8; k++)
      if (x[k] != 0) {
        sum[k] += em[k] - x[k] - g;
        cnt[k]++;
      }
    if (lane == 0) gap[i] = (short)(g == kNoGap ? 0 : g);
  }
#pragma unroll
  for (int k = 0; k < 8; k++) {
    atomicAdd(&sums[32 * k + lane], (unsigned long long)sum[k]);
    atomicAdd(&cnts[32 * k + lane], cnt[k]);
  }
  __syncthreads();
  if (threadIdx.x < n) {
    atomicAdd(&col[threadIdx.x].gaps, sums[threadIdx.x]);
    atomicAdd(&col[threadIdx.x].cnt, cnts[threadIdx.x]);
  }
}

// Digits of a 64 x 64 tile of A into both layouts.  Grid (row tiles up to 128
// rows, column tiles up to 128 columns); zeros beyond m and n.
__global__ void __launch_bounds__(256)
    tc_slice_kernel(const double *__restrict__ A, int64_t lda, int64_t m, int n,
                    const TcCol *__restrict__ col, const short *__restrict__ gap,
                    unsigned char *__restrict__ P1, unsigned char *__restrict__ P2, int nkc,
                    int64_t nic) {
  __shared__ long long q[64][65];
  const int64_t it = blockIdx.x;  // 64-row tile
  const int jt = blockIdx.y;      // 64-column tile
  for (int t = threadIdx.x; t < 4096; t += 256) {
    const int r = t >> 6, c = t & 63;
    const int64_t i = it * 64 + r;
    const int j = jt * 64 + c;
    q[r][c] = (i < m && j < n) ? tc_fix(__ldcs(A + i * lda + j), col[j].emax - 1022 - gap[i]) : 0;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 1024; t += 256) {
    const bool second = t >= 512;  // second layout: rows j, columns i
    const int r = (t & 511) >> 3, g = t & 7;
    if (!second && jt >= nkc) continue;
    uint4 w[kS];
    unsigned *wp = reinterpret_cast<unsigned *>(w);
#pragma unroll
    for (int h = 0; h < 4; h++) {
      long long q0 = second ? q[8 * g + 2 * h][r] : q[r][8 * g + 2 * h];
      long long q1 = second ? q[8 * g + 2 * h + 1][r] : q[r][8 * g + 2 * h + 1];
      unsigned d[kS];
      tc_digits(q0, q1, d);
#pragma unroll
      for (int s = 0; s < kS; s++) wp[4 * s + h] = d[s];
    }
    unsigned char *base;
    int row;
    if (!second) {
      const TcCols tc = tc_cols(n);
      row = (int)(it & 1) * 64 + r;
      base = P1 + ((it >> 1) * tc.tiles + jt * kS) * (int64_t)kPTile;
      if (jt == nkc - 1 && tc.dpt > 1) {
        if (8 * g < 16 * tc.ks)
#pragma unroll
          for (int s = 0; s < kS; s++)
            *reinterpret_cast<uint4 *>(base + (size_t)(s / tc.dpt) * kPTile +
                                       tc_off(row, s % tc.dpt * 16 * tc.ks + 8 * g)) = w[s];
        continue;
      }
    } else {
      row = (jt & 1) * 64 + r;
      base = P2 + ((int64_t)(jt >> 1) * nic + it) * (int64_t)(kS * kPTile);
    }
#pragma unroll
    for (int s = 0; s < kS; s++)
      *reinterpret_cast<uint4 *>(base + (size_t)s * kPTile + tc_off(row, 8 * g)) = w[s];
  }
}

// Digits of v_jc = 2^E_j z_jc for vector c = blockIdx.x (zeros beyond k and n)
// and its exponent F_c (kTcBad: z is not finite).
__global__ void __launch_bounds__(256)
    tc_zprep_kernel(const double *__restrict__ Z, int n, int k, int nv, int nkc,
                    const TcCol *__restrict__ col, unsigned char *__restrict__ Q,
                    int *__restrict__ F, int *__restrict__ ybits, const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  __shared__ int emax[8];
  const int c = blockIdx.x, j = threadIdx.x, lane = j & 31, warp = j >> 5;
  const double z = (c < k && j < n) ? Z[(size_t)c * n + j] : 0.0;
  const int E = j < n ? col[j].emax - 1022 : 0;
  const int ez = (__double2hiint(z) >> 20) & 0x7ff;
  // |v| < 2^(ez - 1022 + E); non-finite z: a marker above every exponent
  int e = ez == 0 ? -100000 : ez == 0x7ff ? 100000 : ez - 1022 + E;
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) emax[warp] = e;
  __syncthreads();
  e = emax[0];
  for (int w = 1; w < 8; w++) e = max(e, emax[w]);
  const bool bad = e >= 100000;
  if (e <= -100000 || bad) e = 0;
  long long q = 0;
  if (ez != 0 && !bad) q = tc_fix(z, e - E);
  if (j == 0) {
    F[c] = bad ? kTcBad : e;
    ybits[c] = kNoBits;
  }
  if (j < nkc * 64) {
    unsigned char *base = Q + (size_t)(j >> 6) * tc_qset(nv) + tc_off(c, j & 63);
    unsigned d[kS];
    tc_digits(q, 0, d);
#pragma unroll
    for (int s = 0; s < kS; s++)
      *reinterpret_cast<unsigned short *>(base + (size_t)s * nv * 128) = (unsigned short)d[s];
  }
}

// ---- tcgen05 ---------------------------------------------------------------

__device__ __forceinline__ unsigned tc_smem(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// K-major tile, rows of 128 bytes, 128-byte swizzle: groups of 8 rows 1024
// bytes apart (descriptor version 1 of this architecture)
constexpr unsigned kTcDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint64_t tc_desc(unsigned lo) {  // lo: address / 16
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(kTcDescHi));
  return d;
}
__device__ __forceinline__ void tc_mma(unsigned d, uint64_t a, uint64_t b, unsigned idesc,
                                       unsigned acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   tc_smem(bar))
               : "memory");
}
__device__ __forceinline__ void tc_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(bar)) : "memory");
}
__device__ __forceinline__ void tc_ld8(unsigned addr, float (&v)[8]) {
  unsigned r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

// a b + c in one instruction (shifts and adds of 64-bit halves take four)
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

struct TcArgs {
  const unsigned char *P, *Q;
  int nkc;               // K chunks of a P row tile
  int tiles;             // STEP 0: row tiles; 1: row tiles of A^T
  int ranges;            // STEP 1: CTAs per row tile, each a range of the chunks
  int n;
  int nv;                // vectors, a multiple of 16
  const short *gap;      // STEP 0: the rows' gaps
  int *ybits;            // STEP 0: bits of the largest |y| 2^(-2 gap) per vector
  int ysh;               // STEP 0, W = 8: Y in units of 2^(F_c - 54 - ysh)
  long long *Y;          // STEP 0: y, vector c at c ldy
  int64_t ldy;
  long long *H;          // STEP 1: partial sums [range][nv][lo, hi][128 tiles]
  const DevState *gate;
  int *err;
};

// STEP 0: y (P = A), one accumulation per row tile; STEP 1: h (P = A^T), one
// per kFlushChunks chunks of the CTA's range.  W: the weights kept, t + s < W.
template <int STEP, int W>
__global__ void __launch_bounds__(kTcThreads, 1) tc_gemm_kernel(const TcArgs a) {
  if (a.gate != nullptr && *(volatile const int *)&a.gate->done) return;
  extern __shared__ __align__(1024) unsigned char tsm_raw[];
  __shared__ uint64_t pfull[kPStages], pempty[kPStages], qfull[2], qempty[2], accfull, accempty, drain;
  __shared__ unsigned tmem_sh;
  __shared__ volatile int abort_sh;
  __shared__ int ymax[64];
  unsigned char *tsm = tsm_raw + ((1024 - (tc_smem(tsm_raw) & 1023)) & 1023);
  unsigned char *ring = tsm, *qbuf = tsm + (size_t)kPStages * kPTile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qbytes = tc_qset(a.nv);
  if (threadIdx.x < 64) ymax[threadIdx.x] = kNoBits;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kPStages; i++) {
      mbar_init(pfull + i, 1);
      mbar_init(pempty + i, 1);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(qfull + i, 1);
      mbar_init(qempty + i, 1);
    }
    mbar_init(&accfull, 1);
    mbar_init(&accempty, kTcThreads - 64);
    mbar_init(&drain, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     tc_smem(&tmem_sh))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = tmem_sh;

  // the CTA's accumulations: group g covers chunks [cb, ce) of row tile mt
  int ngroups, c_lo = 0, c_hi = a.nkc, mt0;
  if (STEP == 0) {
    mt0 = blockIdx.x;
    ngroups = mt0 < a.tiles ? (a.tiles - mt0 + gridDim.x - 1) / gridDim.x : 0;
  } else {
    mt0 = blockIdx.x % a.tiles;
    const int rg = blockIdx.x / a.tiles, per = (a.nkc + a.ranges - 1) / a.ranges;
    c_lo = min(a.nkc, rg * per);
    c_hi = min(a.nkc, c_lo + per);
    ngroups = (c_hi - c_lo + kFlushChunks - 1) / kFlushChunks;
  }
  auto group = [&](int g, int &mt, int &cb, int &ce) {
    if (STEP == 0) {
      mt = mt0 + g * gridDim.x;
      cb = 0;
      ce = a.nkc;
    } else {
      mt = mt0;
      cb = c_lo + g * kFlushChunks;
      ce = min(c_hi, cb + kFlushChunks);
    }
  };
  const TcCols cols = tc_cols(a.n);
  // a wait that gives up when its limit runs out or another role has
  auto wait = [&](uint64_t *bar, unsigned phase) {
    if (mbar_try_wait(bar, phase)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, phase)) {
      if (abort_sh) return false;
      if (global_ns() - t0 > kTcWaitNs) {
        abort_sh = 1;
        if (a.err != nullptr) atomicCAS(a.err, 0, (int)LSQ_ERR_TIMEOUT);
        return false;
      }
    }
    return true;
  };

  if (warp == 0 && lane == 0) {
    // producer
    const uint64_t pol = l2_evict_first(), polq = l2_evict_last();
    int ps = 0, qs = 0;
    unsigned pph = 0, qph = 0;
    int pn = 0, qn = 0;  // copies issued
    bool ok = true;
    for (int g = 0; g < ngroups && ok; g++) {
      int mt, cb, ce;
      group(g, mt, cb, ce);
      for (int c = cb; c < ce && ok; c++) {
        if (!(ok = wait(qempty + qs, qph ^ 1u))) break;
        mbar_expect_tx(qfull + qs, qbytes);
        bulk_g2s(qbuf + (size_t)qs * qbytes, a.Q + (size_t)c * qbytes, qbytes, qfull + qs, polq);
        qn++;
        if (++qs == 2) {
          qs = 0;
          qph ^= 1u;
        }
        // STEP 1: the rows beyond n of the last row tile are not copied (what
        // they hold reaches only sums that nothing reads)
        const unsigned char *pb =
            STEP == 0 ? a.P + ((int64_t)mt * cols.tiles + c * kS) * (int64_t)kPTile
                      : a.P + ((int64_t)mt * a.nkc + c) * (int64_t)(kS * kPTile);
        const int nt = STEP == 0 && c == a.nkc - 1 ? cols.tiles - c * kS : kS;
        const unsigned bytes = STEP == 0 ? kPTile : 1024u * ((min(128, a.n - 128 * mt) + 7) / 8);
        for (int t = 0; t < nt; t++) {
          if (!(ok = wait(pempty + ps, pph ^ 1u))) break;
          mbar_expect_tx(pfull + ps, bytes);
          bulk_g2s(ring + (size_t)ps * kPTile, pb + (size_t)t * kPTile, bytes, pfull + ps, pol);
          pn++;
          if (++ps == kPStages) {
            ps = 0;
            pph ^= 1u;
          }
        }
      }
    }
    // the copies in flight land before the shared memory is released (the
    // last one of every stage; bounded)
    for (int i = 0; i < kPStages && i < pn; i++) {
      const int q = pn - 1 - i;
      mbar_wait(pfull + q % kPStages, (unsigned)((q / kPStages) & 1), kTcWaitNs);
    }
    for (int i = 0; i < 2 && i < qn; i++) {
      const int q = qn - 1 - i;
      mbar_wait(qfull + (q & 1), (unsigned)((q >> 1) & 1), kTcWaitNs);
    }
  } else if (warp == 1 && lane == 0) {
    // issuer: D FP32, A and B bf16, both K-major, M = 128 (N is added per MMA)
    const unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
    const int gq = 256 / a.nv;
    int ps = 0, qs = 0;
    unsigned pph = 0, qph = 0;
    bool ok = true;
    for (int g = 0; g < ngroups && ok; g++) {
      int mt, cb, ce;
      group(g, mt, cb, ce);
      if (!(ok = wait(&accempty, (unsigned)((g & 1) ^ 1)))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int c = cb; c < ce && ok; c++) {
        if (!(ok = wait(qfull + qs, qph))) break;
        const bool last = STEP == 0 && c == a.nkc - 1;
        const int ks = last ? cols.ks : 4, dpt = last ? cols.dpt : 1;  // K steps of 16
        int q = 0;  // digit t's place in its tile
        const unsigned qb = tc_smem(qbuf + (size_t)qs * qbytes) >> 4, qstep = a.nv * 8;
#pragma unroll
        for (int t = 0; t < kS; t++) {
          if (q == 0) {
            if (!(ok = wait(pfull + ps, pph))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const unsigned pb = (tc_smem(ring + (size_t)ps * kPTile) >> 4) + 2 * ks * q;
          // One MMA covers up to gq digits of Q: their tiles follow each other
          // in shared memory and the accumulators t + s, t + s + 1, ... in
          // TMEM, so they are one operand of up to 256 columns (28 MMAs of 64
          // columns per K step ran at a third of the rate)
#pragma unroll
          for (int kk = 0; kk < 4; kk++) {
            if (kk < ks) {
              const unsigned acc = (c > cb || t > 0 || kk > 0) ? 1u : 0u;
              const uint64_t da = tc_desc(pb + 2 * kk);
              const int se = min(kS, W - t);  // digits of Q for this one of P
              // weight 7's accumulator begins with (1, 6), in an MMA of its own
              const int sw = W > kS && t == 1 ? se - 1 : se;
              for (int s = 0; s < sw; s += gq) {
                const unsigned gd = min(gq, sw - s);
                tc_mma(tmem + a.nv * (s + t), da, tc_desc(qb + s * qstep + 2 * kk),
                       idesc | (gd * (a.nv >> 3)) << 17, acc);
              }
              if (sw < se)
                tc_mma(tmem + a.nv * (sw + t), da, tc_desc(qb + sw * qstep + 2 * kk),
                       idesc | (a.nv >> 3) << 17, c > cb || kk > 0 ? 1u : 0u);
            }
          }
          if (++q == dpt || t == kS - 1) {
            q = 0;
            tc_commit(pempty + ps);
            if (++ps == kPStages) {
              ps = 0;
              pph ^= 1u;
            }
          }
        }
        if (!ok) break;
        tc_commit(qempty + qs);
        if (++qs == 2) {
          qs = 0;
          qph ^= 1u;
        }
      }
      if (ok) tc_commit(&accfull);
    }
  } else if (warp >= 2) {
    // four warps per quarter of the 128 lanes; 8 vectors of every 32 each.  The
    // next accumulation waits for the last warp's loads: a warp combines its
    // first 8 vectors (56 registers to 16), loads the second 8, and lets TMEM go
    // before it stores anything
    const int w = warp & 3, row = 32 * w + lane, sub = (warp - 2) >> 2;
    const unsigned tl = tmem + ((unsigned)(32 * w) << 16);
    const size_t ldh = 128 * (size_t)a.tiles;
    for (int g = 0; g < ngroups; g++) {
      int mt, cb, ce;
      group(g, mt, cb, ce);
      const int gap2 = STEP == 0 ? 2 * a.gap[128 * (int64_t)mt + row] : 0;
      // one decision per warp
      if (!__all_sync(0xffffffffu, wait(&accfull, (unsigned)(g & 1)))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float T[W][8];
      long long v0[8];
      int v1[8];  // STEP 1: the high sum
      auto load = [&](int c0) {
#pragma unroll
        for (int d = 0; d < W; d++) tc_ld8(tl + a.nv * d + c0, T[d]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int d = 0; d < W; d++)
#pragma unroll
          for (int e = 0; e < 8; e++)
            asm volatile("" : "+f"(T[d][e])::"memory");  // no use before the wait
      };
      auto release = [&]() {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        tc_arrive(&accempty);
      };
      auto combine = [&]() {
#pragma unroll
        for (int e = 0; e < 8; e++) {
          if (STEP == 0) {
            // y in units of 2^(F_c - 54): sum_d T_d 256^(5 - d); W = 8: ysh bits
            // more, as many as |y| < n 2^F_c leaves room for
            long long y = __float2int_rn(T[5][e]);
            if (W == kS) y += (__float2int_rn(T[6][e]) + 128) >> 8;
            y = mad_wide(__float2int_rn(T[4][e]), 1 << 8, y);
            y = mad_wide(__float2int_rn(T[3][e]), 1 << 16, y);
            y = mad_wide(__float2int_rn(T[2][e]), 1 << 24, y);
            y += (long long)(__float2int_rn(T[1][e]) + (__float2int_rn(T[0][e]) << 8)) << 32;
            if (W > kS) {
              const long long low = mad_wide(__float2int_rn(T[6][e]), 1 << 8,
                                             (long long)__float2int_rn(T[W - 1][e]));
              y = (y << a.ysh) + ((low + (1ll << (15 - a.ysh))) >> (16 - a.ysh));
            }
            v0[e] = y;
          } else {
            // exact in two 64-bit sums: lo = sum_{d >= 2} T_d 256^(6 - d), hi = T_1 +
            // 256 T_0 (A^T r cancels: rounding the sum to 64 bits at 2^-50 of its
            // terms cost the residual pass a factor 100 in backward error); lo's
            // bits from 40 up are hi's units, so lo's sum stays below 2^63 over
            // 2^23 accumulations
            long long lo = __float2int_rn(T[6][e]);
            if (W > kS) lo += (__float2int_rn(T[W - 1][e]) + 128) >> 8;
            lo = mad_wide(__float2int_rn(T[5][e]), 1 << 8, lo);
            lo = mad_wide(__float2int_rn(T[4][e]), 1 << 16, lo);
            lo = mad_wide(__float2int_rn(T[3][e]), 1 << 24, lo);
            lo += (long long)__float2int_rn(T[2][e]) << 32;
            v1[e] =  // |T_1| <= 2^23, |T_0| <= 2^22
                __float2int_rn(T[1][e]) + (__float2int_rn(T[0][e]) << 8) + (int)(lo >> 40);
            v0[e] = lo & ((1ll << 40) - 1);
          }
        }
      };
      auto store = [&](int c0) {
#pragma unroll
        for (int e = 0; e < 8; e++) {
          if (STEP == 0) {
            const long long y = v0[e];
            a.Y[(size_t)(c0 + e) * a.ldy + 128 * (int64_t)mt + row] = y;
            const int bits = __reduce_max_sync(0xffffffffu, 64 - __clzll(y < 0 ? -y : y) - gap2);
            if (lane == 0) atomicMax(&ymax[c0 + e], bits);
          } else {
            // no other thread adds here: integer reductions without a reply
            // (loads and stores cost a round trip each, 80k cycles per flush)
            unsigned long long *p = reinterpret_cast<unsigned long long *>(
                a.H + 2 * ((size_t)(blockIdx.x / a.tiles) * a.nv + c0 + e) * ldh + 128 * mt + row);
            atomicAdd(p, (unsigned long long)v0[e]);
            atomicAdd(p + ldh, (unsigned long long)(long long)v1[e]);
          }
        }
      };
      const int c0 = 8 * sub, c1 = c0 + 32;
      if (c0 < a.nv) {
        load(c0);
        if (c1 >= a.nv) release();
        combine();
        if (c1 < a.nv) {
          load(c1);
          release();
          store(c0);
          combine();
          store(c1);
        } else {
          store(c0);
        }
      } else {
        release();
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (STEP == 0 && threadIdx.x < a.nv) {
    atomicMax(a.ybits + threadIdx.x, ymax[threadIdx.x]);
  }
  if (abort_sh && warp == 1 && lane == 0) {
    // MMAs in flight end before the TMEM is freed (bounded)
    tc_commit(&drain);
    mbar_wait(&drain, 0, kTcWaitNs);
  }
  __syncthreads();
  if (warp == 2)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// The digits of 2^-g_i y_i (Y holds 2^g_i y_i), 55 bits against the vector's
// largest, < 2^ybits: one CTA per 64 rows, a thread 8 rows of one vector (16 bytes
// of a tile row per digit).
__global__ void __launch_bounds__(256)
    tc_yprep_kernel(const long long *__restrict__ Y, int64_t ldy, int nv,
                    const int *__restrict__ ybits, const short *__restrict__ gap,
                    unsigned char *__restrict__ Q, const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  const int64_t ic = blockIdx.x;
  for (int t = threadIdx.x; t < nv * 8; t += 256) {
    const int c = t >> 3, g = t & 7, sh0 = ybits[c] - 55;
    const uint4 gp = *reinterpret_cast<const uint4 *>(gap + ic * 64 + 8 * g);  // 8 gaps, 0 .. 2046
    const unsigned gw[4] = {gp.x, gp.y, gp.z, gp.w};
    const longlong2 *yp = reinterpret_cast<const longlong2 *>(Y + (size_t)c * ldy + ic * 64 + 8 * g);
    uint4 w[kS];
    unsigned *wp = reinterpret_cast<unsigned *>(w);
#pragma unroll
    for (int h = 0; h < 4; h++) {
      const longlong2 v = __ldcs(yp + h);
      long long q0 = shift_round(v.x, sh0 + 2 * (int)(gw[h] & 0xffffu));
      long long q1 = shift_round(v.y, sh0 + 2 * (int)(gw[h] >> 16));
      unsigned d[kS];
      tc_digits(q0, q1, d);
#pragma unroll
      for (int s = 0; s < kS; s++) wp[4 * s + h] = d[s];
    }
    unsigned char *base = Q + (size_t)ic * tc_qset(nv) + tc_off(c, 8 * g);
#pragma unroll
    for (int s = 0; s < kS; s++) *reinterpret_cast<uint4 *>(base + (size_t)s * nv * 128) = w[s];
  }
}

// The residual's middle step, r_i = b_i - (A x)_i per entry in FP64 from Y = 2^g_i
// (A x)_i (in units of 2^(F_c - 54 - ysh)), and 2^-g_i r_i in place of it; partial
// ||r_c||^2 and the largest biased exponent of every vector's 2^-g_i r_i.  A CTA
// takes blocks of 64 rows (b through shared memory: it is row-major, y is vector
// by vector).
constexpr int kRThreads = 256;
__global__ void __launch_bounds__(kRThreads)
    tc_resid_kernel(long long *__restrict__ Y, int64_t ldy, int64_t m, int k,
                    const double *__restrict__ B, int64_t ldb, const int *__restrict__ F,
                    const short *__restrict__ gap, int ysh, int *__restrict__ rexp,
                    double *__restrict__ r2part) {
  __shared__ double sb[64][65];
  __shared__ double r2s[64];
  __shared__ int ex[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = threadIdx.x; c < 64; c += kRThreads) {
    r2s[c] = 0.0;
    ex[c] = 0;
  }
  for (int64_t i0 = (int64_t)blockIdx.x * 64; i0 < ldy; i0 += (int64_t)gridDim.x * 64) {
    __syncthreads();
    for (int t = threadIdx.x; t < 64 * k; t += kRThreads) {
      const int r = t / k, c = t % k;
      sb[r][c] = i0 + r < m ? __ldcs(B + (i0 + r) * ldb + c) : 0.0;
    }
    __syncthreads();
    const int gp[2] = {gap[i0 + lane], gap[i0 + 32 + lane]};
    for (int c = warp; c < k; c += kRThreads / 32) {
      const int f = F[c];
      double s2 = 0.0;
      int e = 0;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int r = 32 * h + lane;
        long long *p = Y + (size_t)c * ldy + i0 + r;
        const int ex = f - 54 - ysh - gp[h] + 1023;  // the unit's biased exponent
        const double sc = f == kTcBad ? __longlong_as_double(0x7ff8000000000000ll)
                          : ex >= 1 && ex <= 2046 ? __longlong_as_double((long long)ex << 52)
                                                  : ldexp(1.0, ex - 1023);
        const double v = i0 + r < m ? fma(-(double)*p, sc, sb[r][c]) : 0.0;
        const double w = scale_down(v, gp[h]);
        *p = __double_as_longlong(w);
        s2 = fma(v, v, s2);
        e = max(e, (__double2hiint(w) >> 20) & 0x7ff);
      }
      s2 = warp_sum(s2);
      e = __reduce_max_sync(0xffffffffu, e);
      if (lane == 0) {
        r2s[c] += s2;
        ex[c] = max(ex[c], e);
      }
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < k; c += kRThreads) {
    r2part[(size_t)blockIdx.x * k + c] = r2s[c];
    atomicMax(rexp + c, ex[c]);
  }
}

// r's digits (as tc_yprep_kernel, from FP64), and r's scale in F and ybits for
// tc_reduce_kernel.
__global__ void __launch_bounds__(256)
    tc_rprep_kernel(const long long *__restrict__ Y, int64_t ldy, int k, int nv,
                    const int *__restrict__ rexp, unsigned char *__restrict__ Q, int *F,
                    int *ybits) {
  const int64_t ic = blockIdx.x;
  if (ic == 0 && threadIdx.x < nv) {
    const int c = threadIdx.x, e = c < k ? rexp[c] : 0;
    F[c] = e == 0x7ff ? kTcBad : 0;
    ybits[c] = e - 1022 + 54;
  }
  for (int t = threadIdx.x; t < nv * 8; t += 256) {
    const int c = t >> 3, g = t & 7, E = (c < k ? rexp[c] : 0) - 1022;
    const double2 *yp = reinterpret_cast<const double2 *>(Y + (size_t)c * ldy + ic * 64 + 8 * g);
    uint4 w[kS];
    unsigned *wp = reinterpret_cast<unsigned *>(w);
#pragma unroll
    for (int h = 0; h < 4; h++) {
      const double2 v = c < k ? __ldcs(yp + h) : make_double2(0.0, 0.0);
      long long q0 = tc_fix(v.x, E), q1 = tc_fix(v.y, E);
      unsigned d[kS];
      tc_digits(q0, q1, d);
#pragma unroll
      for (int s = 0; s < kS; s++) wp[4 * s + h] = d[s];
    }
    unsigned char *base = Q + (size_t)ic * tc_qset(nv) + tc_off(c, 8 * g);
#pragma unroll
    for (int s = 0; s < kS; s++) *reinterpret_cast<uint4 *>(base + (size_t)s * nv * 128) = w[s];
  }
}

// *r2[c] = the sum of the partials, one warp per vector
__global__ void __launch_bounds__(32)
    tc_r2_kernel(const double *__restrict__ r2part, int np, int k, double *__restrict__ r2) {
  double s = 0.0;
  for (int g = threadIdx.x; g < np; g += 32) s += r2part[(size_t)g * k + blockIdx.x];
  s = warp_sum(s);
  if (threadIdx.x == 0) r2[blockIdx.x] = s;
}

// out[c n + j] = scale[j] 2^(E_j + F_c + ybits_c - 116) (lo + 256^5 hi) summed
// over the ranges: one
// warp per 32 entries j and 8 warps per vector's column block, each every 8th
// partial.
__global__ void __launch_bounds__(256)
    tc_reduce_kernel(const long long *__restrict__ H, int ranges, int nv, int ldh, int n,
                     const TcCol *__restrict__ col, const int *__restrict__ F,
                     const int *__restrict__ ybits, const double *__restrict__ scale,
                     double *__restrict__ out, const DevState *gate) {
  if (gate != nullptr && *(volatile const int *)&gate->done) return;
  __shared__ double red[8][33];
  __shared__ long long redh[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.y;
  const int j = blockIdx.x * 32 + lane;
  double s = 0.0;
  long long hi = 0;  // exact; lo's sums are added in FP64
  if (j < n)
    for (int g = warp; g < ranges; g += 8) {
      const long long *p = H + 2 * ((size_t)g * nv + c) * ldh + j;
      s += (double)p[0];
      hi += p[ldh];
    }
  red[warp][lane] = s;
  redh[warp][lane] = hi;
  __syncthreads();
  if (warp == 0 && j < n) {
    s = 0.0;
    hi = 0;
    for (int w = 0; w < 8; w++) {
      s += red[w][lane];
      hi += redh[w][lane];
    }
    s = fma((double)hi, 1099511627776.0, s);  // 256^5
    s = F[c] == kTcBad ? __longlong_as_double(0x7ff8000000000000ll)
                       : ldexp(s, col[j].emax - 1022 + F[c] + ybits[c] - 116);
    out[(size_t)c * n + j] = scale ? scale[j] * s : s;
  }
}

constexpr int kTcResidCtas = 4;  // per SM

int up(int v, int a) { return (v + a - 1) / a * a; }
int64_t up64(int64_t v, int64_t a) { return (v + a - 1) / a * a; }

}  // namespace

TcSizes multi_tc_sizes(int64_t m, int n, int k, int nsm) {
  TcSizes z;
  const int nv = up(k, 16), njt = up(n, 128) / 128;
  const int64_t mp = up64(m, 128);
  z.p1 = (size_t)(mp / 128) * (up(n, 64) / 64) * kS * kPTile;  // any smaller n fits
  z.p2 = (size_t)njt * (mp / 64) * kS * kPTile;
  z.q = (size_t)(up(n, 64) / 64) * tc_qset(nv);
  z.y = (size_t)(mp / 64) * tc_qset(nv);
  z.y64 = sizeof(long long) * (size_t)mp * nv;
  z.r2 = sizeof(double) * (size_t)nsm * kTcResidCtas * k;
  // (nsm / njt) ranges of njt row tiles: at most nsm tiles, for any smaller n too
  z.h = 2 * sizeof(long long) * (size_t)nsm * nv * 128;
  return z;
}

double multi_tc_pass_bytes(int64_t m, int n) {
  const double mp = (double)up64(m, 128);
  // the first layout whole, of the second the rows below n up to 8
  return mp / 128 * tc_cols(n).tiles * kPTile + mp / 64 * kS * 128.0 * up(n, 8);
}

cudaError_t launch_multi_tc_stats(const double *A, int64_t lda, int64_t m, int n, const TcBufs &b,
                                  int nsm, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(b.col, 0, sizeof(TcCol) * (size_t)n, s);
  if (e != cudaSuccess) return e;
  tc_colmax_kernel<<<nsm * 4, 256, 0, s>>>(A, lda, m, n, b.col);
  tc_rowgap_kernel<<<nsm * 4, 256, 0, s>>>(A, lda, m, up64(m, 128), n, b.col, b.gap);
  return cudaGetLastError();
}

cudaError_t launch_multi_tc_prepare(const double *A, int64_t lda, int64_t m, int n, const TcBufs &b,
                                    cudaStream_t s) {
  const int64_t mp = up64(m, 128);
  tc_slice_kernel<<<dim3((unsigned)(mp / 64), up(n, 128) / 64), 256, 0, s>>>(
      A, lda, m, n, b.col, b.gap, b.p1, b.p2, up(n, 64) / 64, mp / 64);
  return cudaGetLastError();
}

bool multi_tc_columns_ok(int n, const TcCol *col, double bits) {
  for (int j = 0; j < n; j++)
    if (col[j].cnt > 0 && (double)col[j].gaps / (double)col[j].cnt > bits) return false;
  return true;
}

namespace {

// bits that |y| < n 2^F_c leaves above 2^62: n <= 256 >> ysh
int tc_ysh(int n) {
  int sh = 0;
  while (sh < 8 && n <= (128 >> sh)) sh++;
  return sh;
}

struct TcShape {
  int nv, nkc, njt, ranges;
  int64_t mp;
  size_t smem;
};

cudaError_t tc_shape(int64_t m, int n, int k, int nsm, TcShape *t) {
  t->nv = up(k, 16);
  t->nkc = up(n, 64) / 64;
  t->njt = up(n, 128) / 128;
  t->ranges = nsm / t->njt;
  t->mp = up64(m, 128);
  t->smem = (size_t)kPStages * kPTile + 2 * (size_t)tc_qset(t->nv) + 1024;
  const void *fn[] = {(const void *)tc_gemm_kernel<0, 7>, (const void *)tc_gemm_kernel<1, 7>,
                      (const void *)tc_gemm_kernel<0, 8>, (const void *)tc_gemm_kernel<1, 8>};
  cudaError_t e = cudaSuccess;
  for (const void *f : fn)
    if (e == cudaSuccess) e = ensure_smem_attr(f, (int)t->smem);
  return e;
}

// y = A z in 64 bits
template <int W>
void tc_step0(const TcShape &t, int n, int k, const double *Z, const TcBufs &b, int nsm,
              const DevState *gate, int *err, cudaStream_t s) {
  tc_zprep_kernel<<<t.nv, 256, 0, s>>>(Z, n, k, t.nv, t.nkc, b.col, b.q, b.F, b.ybits, gate);
  const TcArgs a = {b.p1, b.q, t.nkc, (int)(t.mp / 128), 1, n, t.nv, b.gap, b.ybits, tc_ysh(n), b.y64, t.mp, nullptr,
                    gate, err};
  tc_gemm_kernel<0, W><<<(int)std::min<int64_t>(nsm, t.mp / 128), kTcThreads, t.smem, s>>>(a);
}

// out = scale .* A^T y from y's digits
template <int W>
cudaError_t tc_step1(const TcShape &t, int n, int k, double *out, const double *scale,
                     const TcBufs &b, const DevState *gate, int *err, cudaStream_t s) {
  const TcArgs a = {b.p2, b.y, (int)(t.mp / 64), t.njt, t.ranges, n, t.nv, nullptr, nullptr, 0, nullptr, 0, b.h,
                    gate, err};
  cudaError_t e =
      cudaMemsetAsync(b.h, 0, 2 * sizeof(long long) * (size_t)t.ranges * t.nv * 128 * t.njt, s);
  if (e != cudaSuccess) return e;
  tc_gemm_kernel<1, W><<<t.ranges * t.njt, kTcThreads, t.smem, s>>>(a);
  tc_reduce_kernel<<<dim3(up(n, 32) / 32, k), 256, 0, s>>>(
      b.h, t.ranges, t.nv, 128 * t.njt, n, b.col, b.F, b.ybits, scale, out, gate);
  return cudaGetLastError();
}

}  // namespace

// Measured at 500000 x 200 x 64: y 371 us (405 with 8 reading warps that stored
// before they let TMEM go; 1.5 GB of digits), y's digits 101 us, h 385 us (1.4 GB;
// the MMAs fill TMEM, so neither hides its accumulators' combination), the rest
// 17 us: 0.88 ms per pass against 5.9 ms in double-float.
cudaError_t launch_multi_tc_pass(int64_t m, int n, int k, const double *Z, double *out,
                                 const double *scale, const TcBufs &b, int nsm,
                                 const DevState *gate, int *err, cudaStream_t s) {
  TcShape t;
  const cudaError_t e = tc_shape(m, n, k, nsm, &t);
  if (e != cudaSuccess) return e;
  tc_step0<kS>(t, n, k, Z, b, nsm, gate, err, s);
  tc_yprep_kernel<<<(unsigned)(t.mp / 64), 256, 0, s>>>(b.y64, t.mp, t.nv, b.ybits, b.gap, b.y, gate);
  return tc_step1<kS>(t, n, k, out, scale, b, gate, err, s);
}

cudaError_t launch_multi_tc_resid(int64_t m, int n, int k, const double *B, int64_t ldb,
                                  const double *X, double *out, const double *scale, double *r2,
                                  const TcBufs &b, int nsm, int *err, cudaStream_t s) {
  TcShape t;
  cudaError_t e = tc_shape(m, n, k, nsm, &t);
  if (e == cudaSuccess) e = cudaMemsetAsync(b.ybits + 64, 0, sizeof(int) * 64, s);
  if (e != cudaSuccess) return e;
  tc_step0<kS + 1>(t, n, k, X, b, nsm, nullptr, err, s);
  const int g = (int)std::min<int64_t>((int64_t)nsm * kTcResidCtas, t.mp / 64);
  tc_resid_kernel<<<g, kRThreads, 0, s>>>(b.y64, t.mp, m, k, B, ldb, b.F, b.gap, tc_ysh(n),
                                          b.ybits + 64, b.r2part);
  tc_rprep_kernel<<<(unsigned)(t.mp / 64), 256, 0, s>>>(b.y64, t.mp, k, t.nv, b.ybits + 64, b.y,
                                                       b.F, b.ybits);
  tc_r2_kernel<<<k, 32, 0, s>>>(b.r2part, g, k, r2);
  return tc_step1<kS + 1>(t, n, k, out, scale, b, nullptr, err, s);
}

}  // namespace lsq
