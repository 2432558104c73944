// exp2 in FP64 by table and polynomial (P. T. P. Tang, "Table-driven implementation of the exponential
// function in IEEE floating-point arithmetic", ACM TOMS 15 (1989)), for kernels that the FP64 pipe
// (2 operations per clock per SM) bounds: 9 FP64 operations and one shared-memory read from the
// argument's factors to the result.
#pragma once

#include <cuda_runtime.h>

namespace pttk {

constexpr int FEXP_N = 64;  // table entries 2^(j / 64)

// Fills the block's table (one entry per thread of the first FEXP_N; the caller synchronises).
__device__ __forceinline__ void fexp_fill(double* tab) {
  for (int j = threadIdx.x; j < FEXP_N; j += blockDim.x) tab[j] = exp2((double)j / FEXP_N);
}

// 2^(x s / 64) for |x s| <= 64 * 1020 (the caller keeps the range). x s is never rounded by itself: k is
// the integer nearest to it, f = x s - k (|f| <= 1/2) comes from one fused multiply-add, and 2^(f/64) - 1 from its
// Taylor series to degree 5 (the first term left out is below 4e-17).
__device__ __forceinline__ double fexp2_64(double x, double s, const double* __restrict__ tab) {
  constexpr double M = 6755399441055744.0;  // 1.5 * 2^52: the sum's low word is the integer
  constexpr double L = 0.010830424696249145;  // ln 2 / 64
  const double z = fma(x, s, M);
  const int k = __double2loint(z);
  const double f = fma(x, s, -(z - M));
  double p = fma(L * L * L * L * L / 120.0, f, L * L * L * L / 24.0);
  p = fma(p, f, L * L * L / 6.0);
  p = fma(p, f, L * L / 2.0);
  p = fma(p, f, L);
  p *= f;
  const double t = tab[k & (FEXP_N - 1)];
  const double r = fma(t, p, t);
  return __hiloint2double(__double2hiint(r) + ((k >> 6) << 20), __double2loint(r));
}

// exp(-a) for a >= 0 or NaN: the table form below 700 (told by the high word: an FP64 comparison would take
// the same pipe), CUDA's exp beyond.
__device__ __forceinline__ double fexp_neg(double a, const double* __restrict__ tab) {
  if ((unsigned)__double2hiint(a) >= 0x4085e000u) return exp(-a);
  return fexp2_64(a, -92.332482616893656768, tab);  // -64 log2(e)
}

}  // namespace pttk
