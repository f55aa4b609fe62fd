// Double-single arithmetic: a value as the unevaluated sum of two FP32 values,
// about 48 significant bits, from error-free transformations: Knuth's TwoSum,
// Dekker's Fast2Sum (|a| >= |b|), and the product of two FP32 values with its
// exact error from one FMA (Ogita, Rump and Oishi, 2005).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace lbm {
namespace {

struct ds {
  float hi, lo;
};

__device__ __forceinline__ ds ds_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ ds ds_fast_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ ds ds_add(ds x, ds y) {
  const ds s = ds_two_sum(x.hi, y.hi);
  return ds_fast_two_sum(s.hi, s.lo + (x.lo + y.lo));
}
__device__ __forceinline__ ds ds_neg(ds x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ ds ds_sub(ds x, ds y) { return ds_add(x, ds_neg(y)); }
__device__ __forceinline__ ds ds_mul(ds x, ds y) {
  const float p = x.hi * y.hi;
  const float e = fmaf(x.hi, y.hi, -p);
  return ds_fast_two_sum(p, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e)));
}
// x times a power of two c (exact, barring overflow and underflow)
__device__ __forceinline__ ds ds_scale_pow2(ds x, float c) { return {x.hi * c, x.lo * c}; }
__device__ __forceinline__ double ds_to_double(ds x) { return (double)x.hi + (double)x.lo; }
// Host and device: the pair nearest to v (|lo| <= ulp(hi)/2).
__host__ __device__ __forceinline__ ds ds_from_double(double v) {
  const float hi = (float)v;
  return {hi, (float)(v - (double)hi)};
}
// An int64 value in units 2^-sc (sc = 58 or 63, |v| < 2^62), to ~48 bits.
// 64-bit integer conversions issue at the FP64 rate on GB300, so v is cut
// into three 21-bit pieces, each converted exactly as a 32-bit integer, and
// the pieces are summed as pairs.
__device__ __forceinline__ ds ds_from_fixed(int64_t v, int sc) {
  const float a = (float)(int32_t)(v >> 42) * 0x1p42f;                 // exact
  const float b = (float)(int32_t)((v >> 21) & 0x1FFFFF) * 0x1p21f;    // exact
  const float c = (float)(int32_t)(v & 0x1FFFFF);                      // exact
  const ds ab = ds_two_sum(a, b);
  const ds r = ds_add(ab, ds{c, 0.f});
  const float scale = sc == 58 ? 0x1p-58f : 0x1p-63f;   // exact: powers of two
  return {r.hi * scale, r.lo * scale};
}

}  // namespace
}  // namespace lbm
