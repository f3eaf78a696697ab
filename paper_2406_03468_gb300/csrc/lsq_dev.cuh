// Device helpers shared by the passes over A and over its FP32 planes
// (lsq_dfpass.cuh, k_multi_df.cu, k_multi_tc.cu and others): error-free FP32
// arithmetic (TwoSum, exact widening to FP64, packed f32x2 double-float steps),
// programmatic dependent launches, sums of partials, mbarrier operations and TMA
// bulk copies.  Internal to liblsq; nothing here is part of the ABI.
#pragma once

#include <stdint.h>

#include "lsq_common.cuh"

namespace lsq {

// Programmatic dependent launch: let the next kernel of the stream take its
// slots, and wait until the previous ones have completed (a no-op in a
// kernel that was launched without the attribute).
__device__ __forceinline__ void griddep_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void griddep_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// A load that stays on its side of griddep_wait: the compiler may move an
// ordinary read-only load down to its first use.
__device__ __forceinline__ double ld_early(const double *p) {
  double v;
  asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
// Launch as a programmatic dependent of the kernel before it in the stream.
// Such a kernel calls griddep_wait before it touches anything that an
// earlier kernel of the chain writes, or that an earlier one still reads.
// What the kernels before it write is not read through the read-only path
// (const __restrict__ parameters, __ldg): it is written after this kernel began.
template <typename... K, typename... T>
cudaError_t launch_pdl(void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       T... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

// Sums over g < grid of part[g npad + j] for the 8 columns j0 .. j0 + 7, by a CTA
// of 256 threads: 32 threads per column take every 32nd partial, then
// shuffles and shared memory (a fixed order).  Column j0 + t on thread t < 8.
constexpr int kReduceThreads = 256;
constexpr int kReduceCols = 8;
__device__ __forceinline__ double sum_partials(const double *part, int grid, int npad, int j0,
                                               double (*red)[kReduceCols]) {
  constexpr int kGroups = kReduceThreads / kReduceCols;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = threadIdx.x % kReduceCols, j = j0 + c;  // < npad
  double s0 = 0.0, s1 = 0.0;
  int g = threadIdx.x / kReduceCols;
#pragma unroll 4
  for (; g + kGroups < grid; g += 2 * kGroups) {
    s0 += part[(size_t)g * npad + j];
    s1 += part[(size_t)(g + kGroups) * npad + j];
  }
  if (g < grid) s0 += part[(size_t)g * npad + j];
  double s = s0 + s1;
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  if (lane < kReduceCols) red[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
    const int q = lane >> 3;
    s = red[q][c] + red[q + 4][c];
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
  }
  return s;
}

// Knuth's TwoSum: s + e = a + b exactly.
__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Exact FP32 -> FP64 widening with integer operations (normal and zero
// inputs; infinities and NaN give NaN or an infinity).
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned e = (b >> 23) & 0xffu;
  if (e == 0) return 0.0;
  const unsigned hw = (b & 0x80000000u) | ((e == 255u ? 2047u : e + 896u) << 20) | ((b & 0x7fffffu) >> 3);
  return __hiloint2double((int)hw, (int)(b << 29));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(bar)),
               "r"(count)
               : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned phase) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"((unsigned)__cvta_generic_to_shared(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase; false after limit_ns.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned phase, uint64_t limit_ns) {
  if (mbar_try_wait(bar, phase)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, phase))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}

// L2 policy for data read once (the planes of A stream through L2 dozens of
// times per solve and would otherwise evict R and the partial sums the small
// kernels between passes read).
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// The opposite: planes that fit in L2 are read dozens of times per solve.
__device__ __forceinline__ uint64_t l2_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// An FP64 value as hi + lo FP32 words (as split_rn), NaN when it is beyond
// FP32's range: a conversion would take an FP64 instruction of 64 cycles.
__device__ __forceinline__ void split_f32x2(double a, float &hi, float &lo) {
  split_rn(a, hi, lo);
  if ((((unsigned)__double2hiint(a) >> 20) & 0x7ffu) >= 896u + 254u) hi = __uint_as_float(0x7fffffffu);
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, unsigned bytes, uint64_t *bar,
                                         uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1], %2, [%3], %4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
      "l"(src), "r"(bytes), "r"((unsigned)__cvta_generic_to_shared(bar)), "l"(pol)
      : "memory");
}

// Packed FP32 pairs (two columns per 64-bit register, the lower one in the
// low word): sm_100-class add / sub / mul / fma .rn.f32x2 round each half as
// the scalar instruction would, at one issue slot per two elements.
typedef unsigned long long f2_t;
__device__ __forceinline__ f2_t f2_add(f2_t a, f2_t b) {
  f2_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t f2_sub(f2_t a, f2_t b) {
  f2_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t f2_mul(f2_t a, f2_t b) {
  f2_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t f2_fma(f2_t a, f2_t b, f2_t c) {
  f2_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2_t f2_pack(float lo, float hi) {
  return ((f2_t)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float f2_lo(f2_t v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2_hi(f2_t v) { return __uint_as_float((unsigned)(v >> 32)); }
// One double-float accumulation step on a pair: (s, l) += (a * b exactly,
// with the cross terms a * bl + al * b), given bn = -b.  The product's
// rounding error comes from fma(a, b, -p) with -p = a * bn; the TwoSum adds p
// as s - (-p).  Every operation is the scalar algorithm's, per half.
__device__ __forceinline__ void f2_dd_step(f2_t &s, f2_t &l, f2_t a, f2_t al, f2_t b, f2_t bl,
                                           f2_t bn) {
  const f2_t pn = f2_mul(a, bn);
  const f2_t c = f2_fma(a, bl, f2_fma(al, b, f2_fma(a, b, pn)));
  const f2_t s1 = f2_sub(s, pn);
  const f2_t bb = f2_sub(s1, s);
  const f2_t er = f2_sub(f2_sub(s, f2_sub(s1, bb)), f2_add(pn, bb));
  s = s1;
  l = f2_add(l, f2_add(er, c));
}

// Renormalisation of a packed double-float pair by TwoSum (exact whatever
// the magnitudes): (s, l) <- (fl(s + l), the exact remainder).
__device__ __forceinline__ void f2_renorm(f2_t &s, f2_t &l) {
  const f2_t t = f2_add(s, l);
  const f2_t bb = f2_sub(t, s);
  l = f2_add(f2_sub(s, f2_sub(t, bb)), f2_sub(l, bb));
  s = t;
}

}  // namespace lsq
