// Double-float ("df") arithmetic on the FP32 pipe.
//
// A df value is an unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// i.e. a 48-bit significand.  On this GPU the FP64 pipe issues about 1/64 of the
// FP32 rate, so the recurrences of the mixed path that need more than FP32
// (the ion state update and the spectral y-eliminations of the ill-conditioned
// low wavenumbers) run in df instead of FP64.  Building blocks: Knuth's
// error-free TwoSum, Dekker's FastTwoSum and the FMA form of Dekker's TwoProduct
// (Dekker 1971; Knuth, TAOCP vol. 2, 4.2.2).  Every operation uses the
// explicitly rounded intrinsics so that the compiler cannot contract a
// product and a sum into an FMA, which would break the error-free transforms.
#pragma once

#include <cuda_runtime.h>

namespace pnp {

struct dfl {
  float h, l;
};

// s + e == a + b exactly, s = fl(a + b).
__device__ __forceinline__ dfl df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

// Same, valid when |a| >= |b| (or a == 0).
__device__ __forceinline__ dfl df_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// a * b for df operands; the lo * lo term is below the df resolution.
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return df_fast_two_sum(p, e);
}

// x + a * b as one step of a recurrence in b: the product's trailing part is not
// normalised before the sum, and the sum once, by FastTwoSum.  Error about 2^-47 (|x| +
// |a b|), as with the parts normalised one by one; after a cancellation what FastTwoSum
// drops is a rounding of the trailing part, 2^-48 of the operands.  Eight dependent
// operations from b to the result's leading part, against 23.  A whole elimination's rms
// error against 80-bit arithmetic, relative to its column's largest value, with the
// parts normalised one by one and so: 6.0e-15 and 5.4e-15 at 64 rows (1.3e-15 and
// 1.2e-15 between Dirichlet walls), 3.3e-14 and 3.0e-14 at 192 (1.6e-15 and 2.0e-15),
// 2.9e-13 both at 384: it goes either way, 1e-5 of the rounding of the FP32 solution
// that is stored (8e-9).
__device__ __forceinline__ dfl df_add_mul(dfl x, dfl a, dfl b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  const dfl s = df_two_sum(x.h, p);
  const float lo = __fadd_rn(s.l, __fadd_rn(x.l, e)), h = __fadd_rn(s.h, lo);
  return {h, __fsub_rn(lo, __fsub_rn(h, s.h))};
}

// x + d + f with x, d df and f a float; renormalised with TwoSum because the
// leading sum may cancel.
__device__ __forceinline__ dfl df_add2(dfl x, dfl d, float f) {
  const dfl s1 = df_two_sum(x.h, d.h);
  const dfl s2 = df_two_sum(s1.h, f);
  const float t = __fadd_rn(__fadd_rn(x.l, d.l), __fadd_rn(s1.l, s2.l));
  return df_two_sum(s2.h, t);
}

// x + y for df operands, with both the leading and the trailing parts summed
// by TwoSum (the accurate df sum: valid when x and y have opposite signs and
// cancel).
__device__ __forceinline__ dfl df_add(dfl x, dfl y) {
  dfl s = df_two_sum(x.h, y.h);
  const dfl t = df_two_sum(x.l, y.l);
  s = df_fast_two_sum(s.h, __fadd_rn(s.l, t.h));
  return df_fast_two_sum(s.h, __fadd_rn(s.l, t.l));
}

// x + y for df operands with the trailing parts added in FP32 (Dekker's
// sum): error about 2^-47 (|x| + |y|), enough for running sums whose terms do
// not cancel to far below their own size.
__device__ __forceinline__ dfl df_add_fast(dfl x, dfl y) {
  const dfl s = df_two_sum(x.h, y.h);
  return df_fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}

// a * b exactly, for float operands (TwoProduct).
__device__ __forceinline__ dfl df_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}

// Two df values side by side (the real and imaginary part of a complex value) in
// packed FP32: the same operations in the same order as above, so each lane
// equals the scalar result bit for bit (a - b as fma(b, -1, a): one rounding).
struct df2 {
  float2 h, l;
};
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }
__device__ __forceinline__ df2 df2_two_sum(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  const float2 bb = sub2(s, a);
  return {s, __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ df2 df2_mul(df2 a, dfl b) {
  const float2 bh = f2(b.h), p = __fmul2_rn(a.h, bh);
  float2 e = __ffma2_rn(a.h, bh, __fmul2_rn(p, f2(-1.f)));
  e = __ffma2_rn(a.h, f2(b.l), e);
  e = __ffma2_rn(a.l, bh, e);
  const float2 s = __fadd2_rn(p, e);
  return {s, sub2(e, sub2(s, p))};
}
__device__ __forceinline__ df2 df2_add_mul(df2 x, dfl a, df2 b) {
  const float2 ah = f2(a.h), p = __fmul2_rn(ah, b.h);
  float2 e = __ffma2_rn(ah, b.h, __fmul2_rn(p, f2(-1.f)));
  e = __ffma2_rn(ah, b.l, e);
  e = __ffma2_rn(f2(a.l), b.h, e);
  const df2 s = df2_two_sum(x.h, p);
  const float2 lo = __fadd2_rn(s.l, __fadd2_rn(x.l, e)), h = __fadd2_rn(s.h, lo);
  return {h, sub2(lo, sub2(h, s.h))};
}

// Host-side split of a double into a df pair (hi = nearest float).
inline dfl df_split_host(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

}  // namespace pnp
