// Double-float arithmetic of the mixed mode: a value as an unevaluated sum
// hi + lo of two FP32 numbers.  Sums use Knuth's error-free TwoSum (the rounding
// error of a + b is exactly representable and recovered with six additions)
// accumulated as in the cascaded summation of Ogita, Rump and Oishi (SIAM J.
// Sci. Comput. 26, 2005); products use the FMA-based exact product.  The result
// is as accurate as a sum evaluated in twice the FP32 precision and then
// rounded — ample for momentum sums rounded to FP32 and for k^2 - m^2 near a
// pole — while GB300 runs FP32 at 64 times its FP64 rate.
// The error terms are those of the rounded products and sums, so these are
// written with the intrinsics that the compiler does not contract: a + b c as
// one FMA would leave the rounding error of b c out of the sum, and the low part
// would then count it once more.
#pragma once

namespace mg {

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

struct dfl {
  float hi, lo;
};
__device__ __forceinline__ dfl two_sum(float a, float b) {
  const float s = add_rn(a, b), bb = add_rn(s, -a);
  return {s, add_rn(add_rn(a, -add_rn(s, -bb)), add_rn(b, -bb))};
}
__device__ __forceinline__ dfl dfl_split(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
// sum of signed terms t_k = hi_k + lo_k, k = 0..n-1 (V: float, or a pair of events)
template <class V>
struct DflSum {
  V s, err;
  __device__ __forceinline__ void first(V hi, V lo) { s = hi; err = lo; }
  __device__ __forceinline__ void add(V hi, V lo) {
    const V t = add_rn(s, hi), b = add_rn(t, -s);
    err = err + (add_rn(add_rn(s, -add_rn(t, -b)), add_rn(hi, -b)) + lo);
    s = t;
  }
  __device__ __forceinline__ V value() const { return s + err; }
};

// k^2 of a double-float four-vector from the exact squares of the components
template <class V>
__device__ __forceinline__ DflSum<V> dfl_invariant(const DflSum<V>* k) {
  DflSum<V> d;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const V h = k[mu].s, p = mul_rn(h, h);
    const V e = fmac(V(2.0f) * h, k[mu].err, fmac(h, h, -p));
    if (mu == 0) d.first(p, e);
    else d.add(-p, -e);
  }
  return d;
}

// Products, sums, reciprocals and reciprocal square roots of double-floats (the
// low parts not normalised), accurate to a few 2^-46.
__device__ __forceinline__ dfl dfl_mul(dfl a, dfl b) {
  const float p = mul_rn(a.hi, b.hi);
  return {p, fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, fmaf(a.hi, b.hi, -p)))};
}
__device__ __forceinline__ dfl dfl_add(dfl a, dfl b) {
  const dfl s = two_sum(a.hi, b.hi);
  return {s.hi, s.lo + (a.lo + b.lo)};
}
__device__ __forceinline__ float dfl_value(dfl a) { return a.hi + a.lo; }
// one Newton step in FP32 on the FP32 value, its residual formed with FMAs; a
// residual that is not small (the square of the value overflows) is dropped
__device__ __forceinline__ float small_or_zero(float r) { return fabsf(r) < 1e-3f ? r : 0.0f; }
__device__ __forceinline__ dfl dfl_rsqrt(dfl s) {
  const float y = rsqrtf(s.hi), t = mul_rn(y, y), tl = fmaf(y, y, -t);
  const float r = fmaf(s.hi, t, -1.0f) + fmaf(s.hi, tl, s.lo * t);
  return {y, -0.5f * y * small_or_zero(r)};
}
__device__ __forceinline__ dfl dfl_rcp(dfl b) {
  const float y = 1.0f / b.hi;
  return {y, y * small_or_zero(-fmaf(b.hi, y, -1.0f) - b.lo * y)};
}

}  // namespace mg
