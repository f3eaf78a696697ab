// The inner pass over the FP32 planes of A, shared by the plans' kernels
// (k_pass_df.cu) and the batched engine (k_batch.cu):
//
//   MODE 0  h = A^T (A z) in double-float on the hi / lo planes: t_i = sum_j
//           a_ij z_j by TwoProd of hi * z_hi, the cross terms hi * z_lo and
//           lo * z_hi added to the error word, TwoSum accumulation; h_j +=
//           a_ij t_i the same way against t = t_hi + t_lo, each column a
//           double-float accumulator flushed into an FP64 one every kDfFlush
//           rows (its error word gathers at most kDfFlush rows of error terms,
//           a relative error of about 2^-43 of the sums; a flush is 4 P FP64
//           warp instructions of 64 cycles)
//   MODE 1  LSQR's pass: r = bscale s - A z, s <- r, sums of A^T r (double-
//           float) and ||r||^2 (FP64); the row result and r are FP64
//   MODE 2  MODE 0 in FP32 on the hi plane (the mixed-precision tier): FP32
//           products and column sums, flushed into FP64 every kDfFlush rows
//
// Tile.  G lanes share a row and hold P pairs of its columns each (packed
// f32x2: two columns per 64-bit register), so 2 G P >= n columns and a warp
// takes 32 / G rows at a time.  G is the smallest of 8, 16, 32 with P <= 8
// (df_tile): the row product's reduction is log2 G shuffle steps for 32 / G
// rows at once, and no lane holds columns beyond the next multiple of 2 G.  A
// pass that is not bound by HBM is bound by its arithmetic: per row about 24 P / 2
// packed operations and 11 log2 G for the reduction, over 32 / G rows (400000 x
// 128: FMA pipe 55% busy, issue slots 54%, DRAM 66% of its nominal rate; 200000 x
// 500: 62%, 55%, 78%).  Measured, against one row per warp in tiles of 64, 128, 256,
// 512 or 1024 columns with FP64 conversions of z: 1e6 x 500 592 us (672; 6.76 TB/s,
// the measured copy rate), 120000 x 128 28 us (41); whole iterations 100000 x 257 57
// us (102), 60000 x 600 80 us (157), 100000 x 64 23 us (47), LSQR 200000 x 250 110
// us (146).
//
// Rows reach shared memory by TMA bulk copies (cp.async.bulk with mbarrier
// completion), kStages blocks of consecutive rows per warp in flight (at
// least 2 KB per plane where the rows are shorter); every wait is bounded, and
// on a timeout the kernel records LSQ_ERR_TIMEOUT, waits (bounded) for its
// copies in flight and returns.
#pragma once
#include "lsq_common.cuh"
#include "lsq_dev.cuh"

namespace lsq {

constexpr int kDfFlush = 32;
constexpr int kDfWarps = kPassThreads / 32;
constexpr uint64_t kDfWaitNs = 1000ull * 1000 * 1000;  // 1 s

struct DfTile {
  int G, P;
};
// P steps by 2 above 8 pairs (n > 512): half as many kernels, at most 12% of
// the columns idle.
inline __host__ __device__ DfTile df_tile(int n) {
  if (n <= 128) return {8, (n + 15) / 16};
  if (n <= 256) return {16, (n + 31) / 32};
  if (n <= 512) return {32, (n + 63) / 64};
  return {32, (n + 127) / 128 * 2};
}
constexpr int df_stages(int mode) { return mode == 2 ? 4 : 2; }
constexpr int df_planes(int mode) { return mode == 2 ? 1 : 2; }
// floats of one plane per stage: a row of the largest tile, at least 2 KB
constexpr int df_stage_floats(int P) { return P > 8 ? 64 * P : 512; }
constexpr size_t df_smem(int G, int P, int mode) {
  return (size_t)kDfWarps * 2 * G * P * sizeof(double) +
         (size_t)kDfWarps * df_stages(mode) * df_planes(mode) * df_stage_floats(P) * sizeof(float) +
         (size_t)kDfWarps * df_stages(mode) * sizeof(uint64_t);
}
// rows of one staged block (a multiple of the 32 / G rows a warp takes at once)
inline __host__ __device__ int df_block_rows(DfTile t, int ld32) {
  const int rpw = 32 / t.G;
  if (rpw == 1) return 1;  // n > 256
  // the last row's tile ends within the stage
  return rpw * ((df_stage_floats(t.P) - 2 * t.G * t.P + ld32) / (rpw * ld32));
}

// v = z 2^-fz split into FP32 words hi + lo (to 2^-48 relative and better)
// with integer operations: eb is the biased exponent of the largest |z|, so
// every v is below 1.  A double's conversions and subtractions would take 5
// FP64 instructions of 64 cycles per element and warp.  Words below 2^-115
// are flushed; a non-finite z gives NaN.
__device__ __forceinline__ void split_scaled(double z, int eb, float &hi, float &lo) {
  const unsigned hw = (unsigned)__double2hiint(z), lw = (unsigned)__double2loint(z);
  const int ez = (int)((hw >> 20) & 0x7ffu);
  const int ef = ez > 0 ? ez - eb + 126 : 0;
  const unsigned sign = hw & 0x80000000u;
  const unsigned up = (lw >> 28) & 1u;
  const unsigned m23 = ((hw & 0xfffffu) << 3) | (lw >> 29);
  const unsigned hib = sign | (((unsigned)ef << 23) + m23 + up);
  const int rem = (int)(lw & 0x1fffffffu) - (up ? (1 << 29) : 0);
  // rem 2^(ef - 127 - 52) = (rem 2^-40) 2^(ef - 139)
  const float l = __fmul_rn(__fmul_rn(__int2float_rn(rem), 9.094947017729282e-13f),
                            __int_as_float((ef > 12 ? ef - 12 : 1) << 23));
  hi = ef > 0 ? __uint_as_float(hib) : 0.0f;
  lo = ef > 12 ? __uint_as_float(__float_as_uint(l) ^ sign) : 0.0f;
  if (eb == 0x7ff) hi = __uint_as_float(0x7fffffffu);
}

// One CTA's share of the pass: rows [r0, r1) of the planes (ld32 floats per
// row, a multiple of 4; 16-byte aligned).  part: the CTA's npad sums; s,
// bscale, r2_out: MODE 1.  done: return once *done is set (after the
// previous kernels have ended).  smem: df_smem(P, MODE) bytes, 16-byte
// aligned.  keep: the planes fit in L2 and should stay there.
template <int G, int P, int MODE>
__device__ __forceinline__ void df_pass_body(const float *__restrict__ Ahi,
                                             const float *__restrict__ Alo, int ld32, int64_t r0,
                                             int64_t r1, int n, const double *z, double *s,
                                             const double *bscale, double *part, double *r2_out,
                                             int npad, const int *done, int *err, bool keep,
                                             double *smem) {
  constexpr int kStages = df_stages(MODE), kPlanes = df_planes(MODE), SF = df_stage_floats(P);
  constexpr int RPW = 32 / G;
  __shared__ double wr2[kDfWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = lane % G, grp = lane / G;
  constexpr int kCols = 2 * G * P;
  float *stages = reinterpret_cast<float *>(smem + (size_t)kDfWarps * kCols);
  uint64_t *bars =
      reinterpret_cast<uint64_t *>(stages + (size_t)kDfWarps * kStages * kPlanes * SF);
  float *wst = stages + (size_t)warp * kStages * kPlanes * SF;
  uint64_t *wbar = bars + warp * kStages;
  const int rb = df_block_rows({G, P}, ld32);
  const int nblk = (int)((r1 - r0 + rb - 1) / rb);  // blocks of this CTA, dealt to its warps
  if (lane == 0) {
    for (int st = 0; st < kStages; st++) mbar_init(wbar + st, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // A lane's tile may reach past its row, where z is 0 and the column sums
  // are not read: what lies there must only be finite.  It is the next row
  // (the planes hold finite values everywhere, pads included), an earlier
  // block's, or, past the first block of a stage, memory that no copy has
  // written: zeroed here.
  if (kCols > ld32)
    for (int k = 0; k < kStages; k++) {
      const int64_t q = warp + k * kDfWarps;
      if (q >= nblk) break;
      const int rows = (int)min((int64_t)rb, r1 - r0 - q * rb), w = kCols - ld32;
      for (int t = lane; t < kPlanes * w; t += 32)
        wst[(size_t)(k * kPlanes + t / w) * SF + rows * ld32 + t % w] = 0.0f;
    }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  const uint64_t pol = keep ? l2_evict_last() : l2_evict_first();
  // the warp's k-th block is block warp + k kDfWarps, in stage k % kStages
  auto issue = [&](int q, int stg) {
    if (lane == 0 && q < nblk) {
      const int64_t i0 = r0 + (int64_t)q * rb;
      const unsigned bytes = (unsigned)(min((int64_t)rb, r1 - i0) * ld32 * sizeof(float));
      float *dh = wst + (size_t)stg * kPlanes * SF;
      mbar_expect_tx(wbar + stg, kPlanes * bytes);
      bulk_g2s(dh, Ahi + i0 * ld32, bytes, wbar + stg, pol);
      if (kPlanes == 2) bulk_g2s(dh + SF, Alo + i0 * ld32, bytes, wbar + stg, pol);
    }
  };
  // the planes were complete before the inner loop began: the first rows are
  // on their way while the kernel that forms z ends
#pragma unroll
  for (int k = 0; k < kStages; k++) issue(warp + k * kDfWarps, k);
  double *hw = smem + (size_t)warp * kCols;
  for (int i = lane; i < kCols; i += 32) hw[i] = 0.0;
  griddep_wait();
  if (done != nullptr && *(volatile const int *)done) {
    if (lane == 0)  // the copies in flight land before the CTA's memory is released
      for (int k = 0; k < kStages; k++)
        if (warp + k * kDfWarps < nblk) mbar_wait(wbar + k, 0, kDfWaitNs);
    return;
  }
  // z scaled by a common power of two: eb, the largest biased exponent (every
  // group of lanes holds all columns); 2^fz = 2^(eb - 1022)
  double zr[2 * P];
  int eb = 0;
#pragma unroll
  for (int k = 0; k < P; k++) {
    const int col = 2 * G * k + 2 * gl;
    zr[2 * k] = (col < n) ? z[col] : 0.0;
    zr[2 * k + 1] = (col + 1 < n) ? z[col + 1] : 0.0;
    eb = max(eb, (__double2hiint(zr[2 * k]) >> 20) & 0x7ff);
    eb = max(eb, (__double2hiint(zr[2 * k + 1]) >> 20) & 0x7ff);
  }
  eb = __reduce_max_sync(0xffffffffu, eb);
  const double up = eb > 0 ? ldexp(1.0, eb - 1022) : 1.0;
  const double bs = MODE == 1 ? *bscale * (eb > 0 ? ldexp(1.0, 1022 - eb) : 1.0) : 0.0;
  f2_t zh[P], zl[MODE == 2 ? 1 : P], zn[MODE == 2 ? 1 : P], hh[P], hl[MODE == 2 ? 1 : P];
#pragma unroll
  for (int k = 0; k < P; k++) {
    float h0, l0, h1, l1;
    split_scaled(zr[2 * k], eb, h0, l0);
    split_scaled(zr[2 * k + 1], eb, h1, l1);
    zh[k] = f2_pack(h0, h1);
    hh[k] = 0ull;
    if (MODE != 2) {
      zl[k] = f2_pack(l0, l1);
      zn[k] = f2_pack(-h0, -h1);
      hl[k] = 0ull;
    }
  }
  double r2 = 0.0, pend = 0.0;  // MODE 1: rows' r until the group's lanes are full
  int64_t pend_i = -1;
  int npend = 0, blk = 0;
  auto flush_pend = [&]() {
    if (pend_i >= 0) {
      s[pend_i] = pend * up;
      r2 = fma(pend, pend, r2);
    }
    pend_i = -1;
    npend = 0;
  };
  // Column sums into the warp's FP64 accumulators.  The groups' sums of a
  // column are first added to each other, halving the pairs a lane holds at
  // each step (lanes 16 apart, then 8): TwoSum of the high words, the errors
  // into the low ones.  32 / G times fewer FP64 instructions, and one
  // accumulator per warp and column.
  auto flush = [&]() {
    constexpr int PA = RPW > 1 ? (P + 1) / 2 : P, PB = RPW > 2 ? (PA + 1) / 2 : PA;
    f2_t vh[PA], vl[PA];
    const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
    auto halve = [&](f2_t eh, f2_t el, f2_t oh, f2_t ol, bool odd, int x, f2_t &rh, f2_t &rl) {
      const f2_t sh = __shfl_xor_sync(0xffffffffu, odd ? eh : oh, x);
      const f2_t sl = __shfl_xor_sync(0xffffffffu, odd ? el : ol, x);
      const f2_t kh = odd ? oh : eh, kl = odd ? ol : el;
      const f2_t t = f2_add(kh, sh), bb = f2_sub(t, kh);
      rl = f2_add(f2_add(kl, sl), f2_add(f2_sub(kh, f2_sub(t, bb)), f2_sub(sh, bb)));
      rh = t;
    };
    if (RPW > 1) {
#pragma unroll
      for (int k = 0; k < PA; k++)
        halve(hh[2 * k], MODE == 2 ? 0ull : hl[MODE == 2 ? 0 : 2 * k],
              2 * k + 1 < P ? hh[2 * k + 1 < P ? 2 * k + 1 : 0] : 0ull,
              (MODE != 2 && 2 * k + 1 < P) ? hl[(MODE != 2 && 2 * k + 1 < P) ? 2 * k + 1 : 0] : 0ull,
              h16, 16, vh[k], vl[k]);
    } else {
#pragma unroll
      for (int k = 0; k < PA; k++) {
        vh[k] = hh[k];
        vl[k] = MODE == 2 ? 0ull : hl[MODE == 2 ? 0 : k];
      }
    }
    if (RPW > 2) {
#pragma unroll
      for (int k = 0; k < PB; k++)
        halve(vh[2 * k], vl[2 * k], 2 * k + 1 < PA ? vh[2 * k + 1 < PA ? 2 * k + 1 : 0] : 0ull,
              2 * k + 1 < PA ? vl[2 * k + 1 < PA ? 2 * k + 1 : 0] : 0ull, h8, 8, vh[k], vl[k]);
    }
#pragma unroll
    for (int k = 0; k < PB; k++) {
      int pk = k;  // the pair that this lane holds
      if (RPW > 2) pk = 2 * pk + (h8 ? 1 : 0);
      if (RPW > 1) pk = 2 * pk + (h16 ? 1 : 0);
      const int col = 2 * G * pk + 2 * gl;
      double c0 = widen(f2_lo(vh[k])), c1 = widen(f2_hi(vh[k]));
      if (MODE != 2 || RPW > 1) {
        c0 += widen(f2_lo(vl[k]));
        c1 += widen(f2_hi(vl[k]));
      }
      if (RPW == 1 || pk < P) {
        hw[col] += c0;
        hw[col + 1] += c1;
      }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < P; k++) {
      hh[k] = 0ull;
      if (MODE != 2) hl[k] = 0ull;
    }
  };
  // MODE 1: s of the group's next row, loaded a row ahead
  double sv = 0.0;
  if (MODE == 1 && warp < nblk) {
    const int64_t i = r0 + (int64_t)warp * rb + grp;
    sv = i < r1 ? s[i] : 0.0;
  }
  int stg = 0;
  unsigned ph = 0;
  int qfail = -1;
  for (int q = warp; q < nblk; q += kDfWarps) {
    // one decision per warp: a lane whose wait ran out takes the whole warp
    // to the drain below
    if (!__all_sync(0xffffffffu, mbar_wait(wbar + stg, ph, kDfWaitNs))) {
      qfail = q;
      break;
    }
    const int64_t i0 = r0 + (int64_t)q * rb;
    const int rows = G == 32 ? 1 : (int)min((int64_t)rb, r1 - i0);
    for (int rr = 0; rr < rows; rr += RPW) {
      const int row = rr + grp;
      const bool ok = G == 32 || row < rows;
      const float *rh = wst + (size_t)stg * kPlanes * SF + (size_t)(ok ? row : rr) * ld32 + 2 * gl;
      f2_t ah[P], al[MODE == 2 ? 1 : P];
#pragma unroll
      for (int k = 0; k < P; k++) {
        ah[k] = *reinterpret_cast<const f2_t *>(rh + 2 * G * k);
        if (MODE != 2) al[k] = *reinterpret_cast<const f2_t *>(rh + SF + 2 * G * k);
      }
      if (G != 32 && !ok) {  // a group beyond the last row adds nothing
#pragma unroll
        for (int k = 0; k < P; k++) {
          ah[k] = 0ull;
          if (MODE != 2) al[k] = 0ull;
        }
      }
      if (rr + RPW >= rows) {
        // every lane has its values: the stage may be refilled (generic reads
        // before the async-proxy writes of the next copy)
        __syncwarp();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(q + kStages * kDfWarps, stg);
      }
      float th, tl = 0.0f;
      if (MODE == 2) {
        f2_t t2 = 0ull;
#pragma unroll
        for (int k = 0; k < P; k++) t2 = f2_fma(ah[k], zh[k], t2);
        th = __fadd_rn(f2_lo(t2), f2_hi(t2));
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) th = __fadd_rn(th, __shfl_xor_sync(0xffffffffu, th, o));
      } else {
        // two independent double-float accumulators (even / odd column, the
        // halves of one packed pair) halve the dependent TwoSum chain
        f2_t shp = 0ull, slp = 0ull;
#pragma unroll
        for (int k = 0; k < P; k++) f2_dd_step(shp, slp, ah[k], al[k], zh[k], zl[k], zn[k]);
        float sh_, sl_, er;
        two_sum_f(f2_lo(shp), f2_hi(shp), sh_, er);
        sl_ = __fadd_rn(__fadd_rn(f2_lo(slp), f2_hi(slp)), er);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, sh_, o);
          const float ol = __shfl_xor_sync(0xffffffffu, sl_, o);
          float sm;
          two_sum_f(sh_, oh, sm, er);
          sh_ = sm;
          sl_ = __fadd_rn(__fadd_rn(sl_, ol), er);
        }
        if (MODE == 0) {
          // renormalise t (Fast2Sum: |sh_| >= |sl_| after the sums above)
          th = __fadd_rn(sh_, sl_);
          tl = __fsub_rn(sl_, __fsub_rn(th, sh_));
        } else {
          // r' = bs s_i - t' in FP64 (2 FP64 instructions for 32 / G rows)
          const double rp = fma(bs, sv, -(widen(sh_) + widen(sl_)));
          split_f32x2(rp, th, tl);
          if (gl == npend && ok) {
            pend = rp;
            pend_i = i0 + row;
          }
          if (++npend == G) flush_pend();
          const bool last = rr + RPW >= rows;
          const int64_t in = last ? i0 + (int64_t)kDfWarps * rb + grp : i0 + row + RPW;
          sv = (in < r1 && (!last || q + kDfWarps < nblk)) ? s[in] : 0.0;
          if (!ok) th = tl = 0.0f;
        }
      }
      const f2_t th2 = f2_pack(th, th);
      if (MODE == 2) {
#pragma unroll
        for (int k = 0; k < P; k++) hh[k] = f2_fma(ah[k], th2, hh[k]);
      } else {
        // column sums: TwoSum into the high word, error terms into the low
        // word, which only gathers kDfFlush rows of small terms before the
        // FP64 flush and is not renormalised row by row
        const f2_t tl2 = f2_pack(tl, tl), tn2 = f2_pack(-th, -th);
#pragma unroll
        for (int k = 0; k < P; k++) f2_dd_step(hh[k], hl[k], ah[k], al[k], th2, tl2, tn2);
      }
      if (++blk == kDfFlush) {
        blk = 0;
        flush();
      }
    }
    if (++stg == kStages) {
      stg = 0;
      ph ^= 1u;
    }
  }
  if (qfail >= 0) {
    // record the error; let the copies this warp has in flight (the blocks
    // qfail, qfail + kDfWarps, ..., one per stage) land before the CTA's
    // shared memory is released (bounded again)
    if (lane == 0) {
      if (err != nullptr) atomicCAS(err, 0, (int)LSQ_ERR_TIMEOUT);
      for (int k = 0, q = qfail; k < kStages && q < nblk; k++, q += kDfWarps) {
        mbar_wait(wbar + stg, ph, kDfWaitNs);
        if (++stg == kStages) {
          stg = 0;
          ph ^= 1u;
        }
      }
    }
    __syncwarp();
  }
  flush();
  if (MODE == 1) {
    flush_pend();
    r2 = warp_sum(r2);
    if (lane == 0) wr2[warp] = r2;
  }
  __syncthreads();
  // fixed-order sum over the warps of this CTA, scaled back by
  // 2^fz: T threads per column take every T-th of them, then one adds the T
  // sums (the stages' memory, free now, holds them)
  constexpr int T = kCols <= 32 ? 8 : kCols <= 64 ? 4 : kCols <= 128 ? 2 : 1;
  double *tsum = reinterpret_cast<double *>(stages);
  for (int c = threadIdx.x; c < kCols * T; c += kPassThreads) {
    const int col = c % kCols, t = c / kCols;
    double sacc = 0.0;
    for (int w = t; w < kDfWarps; w += T) sacc += smem[(size_t)w * kCols + col];
    if (T == 1) {
      if (col < npad) part[col] = sacc * up;
    } else {
      tsum[c] = sacc;
    }
  }
  if (T > 1) {
    __syncthreads();
    for (int col = threadIdx.x; col < kCols && col < npad; col += kPassThreads) {
      double sacc = 0.0;
#pragma unroll
      for (int t = 0; t < T; t++) sacc += tsum[t * kCols + col];
      part[col] = sacc * up;
    }
  }
  if (MODE == 1 && threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kDfWarps; w++) t += wr2[w];
    *r2_out = t * up * up;
  }
}

}  // namespace lsq
