// FP64 roots, reciprocals and warp sums in fewer holds of the FP64 pipe, which is what the eigensolver's chains wait
// for (an FP64 instruction holds its quarter of the SM for 64 cycles, however few lanes take part).
#pragma once
#include "common.cuh"

namespace cakf {

// sqrt(x) and 1 / sqrt(x) for normal x > 0, and 1 / x for normal x with a normal result (the callers scale their
// operands: a denormal one gives NaN), from the hardware's approximations y (about 20 bits,
// full FP64 exponent range) and one third-order step: with e = 1 - x y^2 the factor 1 + e / 2 + 3 e^2 / 8
// (the binomial series of (1 - e)^(-1/2)), with e = 1 - x y the factor 1 + e + e^2.  Both remainders are
// below 2^-56; all three results are within 2^-51 of CUDA's square root and division.
__device__ __forceinline__ void fast_sqrt(double x, double& sq, double& rs) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y;
  const double e = fma(-g, y, 1.0);
  const double f = e * fma(0.375, e, 0.5);
  sq = fma(g, f, g);
  rs = fma(y, f, y);
}
__device__ __forceinline__ double fast_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// Sum of NV doubles per lane over the warp, in every lane, in integer arithmetic.  A shuffle tree costs 126
// cycles a level here (an FP64 operation holds its quarter of the SM for 64 cycles, however few lanes
// take part), integer instructions about 4; so the mantissas are aligned to the largest exponent as three limbs
// of LB bits (72 or 78 bits in all, 19 or more below the largest value's last place; a value's bits below them are
// dropped), the limbs are summed by redux.sync, and the sum is rounded once: more accurate than the tree.  Non-finite or nearly
// overflowing values take the tree.
template <int NV>
__device__ __forceinline__ double warp_sum_int(const double (&x)[NV]) {
  static_assert(NV == 1 || NV == 4, "limbs of NV * 32 values must fit 31 bits");
  constexpr int LB = NV == 1 ? 26 : 24, GUARD = 3 * LB - 53;
  constexpr unsigned MASK = (1u << LB) - 1u;
  unsigned long long m[NV];
  int ex[NV], sg[NV];
  unsigned emax = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const long long b = __double_as_longlong(x[i]);
    ex[i] = (int)((b >> 52) & 0x7FF);
    sg[i] = (int)(b >> 63);
    m[i] = ex[i] ? ((unsigned long long)b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL : 0ULL;
    emax = max(emax, (unsigned)ex[i]);
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  if (emax > 2000u) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < NV; ++i) t += x[i];
    return warp_sum(t);
  }
  int hi = 0, mid = 0, lo = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int d = (int)emax - ex[i];
    const int h = (int)(m[i] >> min(53 - LB + d, 63));
    const int md = (int)((unsigned)(m[i] >> min(53 - 2 * LB + d, 63)) & MASK);
    const int l = (int)((unsigned)(d >= GUARD ? m[i] >> min(d - GUARD, 63) : m[i] << (GUARD - d)) & MASK);
    hi += (h ^ sg[i]) - sg[i];
    mid += (md ^ sg[i]) - sg[i];
    lo += (l ^ sg[i]) - sg[i];
  }
  hi = __reduce_add_sync(0xffffffffu, hi);
  mid = __reduce_add_sync(0xffffffffu, mid);
  lo = __reduce_add_sync(0xffffffffu, lo);
  // hi 2^(2 LB) + mid 2^LB + lo in units of 2^(emax - 1075 - GUARD), as a 64-bit integer times 2^sh
  const long long T = ((long long)hi << LB) + mid;
  const int sh = max(0, LB + 2 - __clzll(T < 0 ? -T : T));
  const long long X = (T << (LB - sh)) + (lo >> sh);
  const double r = __ll2double_rn(X);
  const long long rb = __double_as_longlong(r);
  const int er = (int)((rb >> 52) & 0x7FF) + (int)emax - 1075 - GUARD + sh;
  if (X == 0 || er <= 0) return 0.0;
  return __longlong_as_double((rb & ~(0x7FFLL << 52)) | ((long long)er << 52));
}

}  // namespace cakf
