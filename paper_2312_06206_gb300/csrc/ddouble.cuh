// ddouble.cuh -- double-double arithmetic for set-up tables (about 2^-100): an
// unevaluated sum hi + lo of two doubles, by error-free two-sum (Knuth) and
// two-product (fused multiply-add).
#pragma once

namespace sadi {
namespace dd {

struct D2 {
  double hi, lo;
};

__device__ __forceinline__ D2 two_sum(double a, double b) {
  const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
  return {s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t))};
}
// |a| >= |b|
__device__ __forceinline__ D2 quick_sum(double a, double b) {
  const double s = __dadd_rn(a, b);
  return {s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ D2 two_prod(double a, double b) {
  const double p = __dmul_rn(a, b);
  return {p, __fma_rn(a, b, -p)};
}
__device__ __forceinline__ D2 add(D2 a, D2 b) {
  const D2 s = two_sum(a.hi, b.hi);
  return quick_sum(s.hi, __dadd_rn(s.lo, __dadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ D2 neg(D2 a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ D2 mul(D2 a, double b) {
  const D2 p = two_prod(a.hi, b);
  return quick_sum(p.hi, __fma_rn(a.lo, b, p.lo));
}
__device__ __forceinline__ D2 mul(D2 a, D2 b) {
  const D2 p = two_prod(a.hi, b.hi);
  return quick_sum(p.hi, __dadd_rn(p.lo, __fma_rn(a.hi, b.lo, __dmul_rn(a.lo, b.hi))));
}
__device__ __forceinline__ D2 div(D2 a, double b) {
  const double q = __ddiv_rn(a.hi, b);
  const D2 r = add(a, neg(two_prod(q, b)));
  return quick_sum(q, __ddiv_rn(r.hi, b));
}

// cos(pi p / q), 0 <= p <= 2 q, q <= 2^20: the angle is reduced to [0, pi/4]
// on the integers, then the Taylor series (13 terms: 0.79^28 / 28! < 2^-104)
__device__ inline D2 cospi(int p, int q) {
  const D2 pi{3.141592653589793116, 1.2246467991473532e-16};
  if (p > q) p = 2 * q - p;
  bool minus = false;
  if (2 * p > q) {
    p = q - p;
    minus = true;
  }
  const bool co = 4 * p <= q;   // else the sine of pi/2 - angle
  const D2 x = co ? div(mul(pi, (double)p), (double)q) : div(mul(pi, (double)(q - 2 * p)), (double)(2 * q));
  const D2 x2 = mul(x, x);
  const int odd = co ? 0 : 1;
  D2 r{1.0, 0.0};
  for (int k = 13; k >= 1; --k) r = add({1.0, 0.0}, neg(mul(x2, div(r, (double)((2 * k - 1 + odd) * (2 * k + odd))))));
  if (!co) r = mul(r, x);
  return minus ? neg(r) : r;
}

}  // namespace dd
}  // namespace sadi
