// vof_df.cuh -- double-float arithmetic (unevaluated sums of two FP32
// numbers, ~48 significant bits) for FP64 arithmetic that decides nothing,
// and the WENO5 face value built on it.
//
// On this part an FP64 instruction occupies an SM partition's FP64 unit as
// long as ~64 FP32 instructions occupy the FP32 units, so a value computed
// with a few dozen FP32 instructions to FP64-like accuracy is far cheaper
// than the same value in FP64.  The error-free transformations are the
// classical ones: TwoSum (Knuth), FastTwoSum (Dekker), TwoProduct with a
// fused multiply-add; the pair operations follow Dekker (1971) and the
// double-double algorithms of Hida, Li & Bailey (QD library paper, 2001),
// restated here.  Conversions between FP64 and pairs are done on the bits
// (integer instructions), not by FP64 conversion instructions.
//
// The file is compiled with -fmad=false: no multiply-add is formed except
// where fmaf() is written, which the error-free transformations rely on.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define VOF_HD __host__ __device__ __forceinline__
#else
#define VOF_HD inline
#endif

namespace vofgb {
namespace df {

struct f2 {
  float hi, lo;
};

VOF_HD uint64_t d_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
VOF_HD double bits_d(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
VOF_HD float bits_f(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}
VOF_HD uint32_t f_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
VOF_HD float fma_f(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return fmaf(a, b, c);
#else
  return std::fmaf(a, b, c);
#endif
}

// The two words of an FP64 value, through an opaque move on the device: masks
// of the 64-bit pattern are recognised as FP64 absolute values and negations,
// which are FP64 instructions.
struct words {
  uint32_t hi, lo;
};
VOF_HD words words_of(double x) {
#ifdef __CUDA_ARCH__
  words w;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(w.lo), "=r"(w.hi) : "d"(x));
  return w;
#else
  const uint64_t b = d_bits(x);
  return {(uint32_t)(b >> 32), (uint32_t)b};
#endif
}

// x * 2^-k as a pair: hi = x with its significand truncated to 24 bits
// (exact in FP32, from the bits; 0 below the normal FP32 range; the caller
// keeps x 2^-k below 2^127), lo = the rest (the 29 bits below, an integer in
// units of x's last place), rounded to 24 bits: |x 2^-k - (hi + lo)| <= 2^-48
// |x 2^-k| (and below 2^-125 for parts under the FP32 normal range).  No FP64
// instruction.
VOF_HD f2 split_scaled(words x, int k) {
  const int e = (int)((x.hi >> 20) & 0x7FF) - 1023 - k + 127;  // FP32 exponent field of x 2^-k
  const uint32_t sg = x.hi & 0x80000000u;
  const uint32_t man = ((x.hi & 0xFFFFFu) << 3) | (x.lo >> 29);
  uint32_t h = ((uint32_t)e << 23) | man;
  uint32_t u = (uint32_t)(e - 52) << 23;  // x's last place, scaled
  if (e <= 0) h = 0u;
  if (e <= 52) u = 0u;
  if (e >= 255) h = u = 0x7F800000u;  // beyond FP32: infinity
  return {bits_f(h | sg), (float)(x.lo & 0x1FFFFFFFu) * bits_f(u | sg)};
}

// FP64 value of the FP32 number f * 2^k (exact; f normal or zero)
VOF_HD double widen_scaled(float f, int k) {
  const uint32_t b = f_bits(f);
  const uint32_t ef = (b >> 23) & 0xFF;
  if (ef == 0) return 0.0;
  const uint64_t d = ((uint64_t)(b & 0x80000000u) << 32) | ((uint64_t)(ef + k - 127 + 1023) << 52) |
                     ((uint64_t)(b & 0x7FFFFFu) << 29);
  return bits_d(d);
}

VOF_HD int rint_i(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)std::lrintf(x);
#endif
}
// FP64 value of the pair (hi + lo) * 2^k (|lo| at most half a last place of
// hi): hi widened exactly, then lo added to the bit pattern as an integer
// number of the sum's FP64 last places, to the nearest (half as large when a
// power of two hi meets a lo of the other sign).  A lo whose last places are out of FP32's
// range (hi below 2^-74) is left out.
VOF_HD double widen_pair(f2 q, int k) {
  const uint64_t h = d_bits(widen_scaled(q.hi, k));
  const int eh = (int)((f_bits(q.hi) >> 23) & 0xFF);
  if (eh == 0 || eh == 255) return bits_d(h);
  // towards larger magnitude when the signs agree
  const float l = bits_f(f_bits(q.lo) ^ (f_bits(q.hi) & 0x80000000u));
  const int es = 52 + 127 - (eh - 127) + ((f_bits(q.hi) & 0x7FFFFFu) == 0 && l < 0.0f ? 1 : 0);
  const float up = es > 254 ? 0.0f : bits_f((uint32_t)es << 23);
  return bits_d(h + (uint64_t)(int64_t)rint_i(l * up));
}

// error-free transformations
VOF_HD f2 two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
VOF_HD f2 fast_two_sum(float a, float b) {  // |a| >= |b| or a = 0
  const float s = a + b;
  return {s, b - (s - a)};
}
VOF_HD f2 two_prod(float a, float b) {
  const float p = a * b;
  return {p, fma_f(a, b, -p)};
}

// pair arithmetic (relative error ~2^-46 without cancellation; the sum's
// error is bounded by ~2^-46 of the operands' magnitudes)
VOF_HD f2 add(f2 x, f2 y) {
  f2 s = two_sum(x.hi, y.hi);
  const f2 t = two_sum(x.lo, y.lo);
  s.lo += t.hi;
  s = fast_two_sum(s.hi, s.lo);
  s.lo += t.lo;
  return fast_two_sum(s.hi, s.lo);
}
// the same in 11 operations instead of 20, the error bounded by ~2^-46 of the
// operands' magnitudes (no bound relative to a cancelled sum)
VOF_HD f2 add_c(f2 x, f2 y) {
  f2 s = two_sum(x.hi, y.hi);
  s.lo += x.lo + y.lo;
  return fast_two_sum(s.hi, s.lo);
}
VOF_HD f2 neg(f2 x) { return {-x.hi, -x.lo}; }
VOF_HD f2 twice(f2 x) { return {2.0f * x.hi, 2.0f * x.lo}; }  // exact
VOF_HD f2 mul(f2 x, f2 y) {
  f2 p = two_prod(x.hi, y.hi);
  p.lo = fma_f(x.hi, y.lo, fma_f(x.lo, y.hi, p.lo));
  return fast_two_sum(p.hi, p.lo);
}
// times a small integer constant (exact in FP32)
VOF_HD f2 mul_k(f2 x, float k) {
  f2 p = two_prod(x.hi, k);
  p.lo = fma_f(x.lo, k, p.lo);
  return fast_two_sum(p.hi, p.lo);
}
VOF_HD f2 sqr(f2 x) {
  f2 p = two_prod(x.hi, x.hi);
  p.lo = fma_f(2.0f * x.hi, x.lo, p.lo);
  return fast_two_sum(p.hi, p.lo);
}

// Two FP32 values side by side: one packed instruction per operation on this
// architecture (the same roundings as two separate ones).
struct v2 {
#ifdef __CUDA_ARCH__
  unsigned long long b;
#else
  float x, y;
#endif
};
VOF_HD v2 vset(float x, float y) {
#ifdef __CUDA_ARCH__
  v2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.b) : "f"(x), "f"(y));
  return r;
#else
  return {x, y};
#endif
}
VOF_HD void vget(v2 a, float& x, float& y) {
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.b));
#else
  x = a.x;
  y = a.y;
#endif
}
VOF_HD v2 vadd(v2 a, v2 b) {
#ifdef __CUDA_ARCH__
  v2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
  return r;
#else
  return {a.x + b.x, a.y + b.y};
#endif
}
VOF_HD v2 vmul(v2 a, v2 b) {
#ifdef __CUDA_ARCH__
  v2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
  return r;
#else
  return {a.x * b.x, a.y * b.y};
#endif
}
VOF_HD v2 vfma(v2 a, v2 b, v2 c) {
#ifdef __CUDA_ARCH__
  v2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(a.b), "l"(b.b), "l"(c.b));
  return r;
#else
  return {std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)};
#endif
}
// a - b as one fused multiply-add: the same rounding
VOF_HD v2 vsub(v2 a, v2 b) { return vfma(b, vset(-1.0f, -1.0f), a); }

// two pairs side by side
struct f2x2 {
  v2 hi, lo;
};
VOF_HD f2x2 both(f2 x, f2 y) { return {vset(x.hi, y.hi), vset(x.lo, y.lo)}; }
VOF_HD void each(f2x2 a, f2& x, f2& y) {
  vget(a.hi, x.hi, y.hi);
  vget(a.lo, x.lo, y.lo);
}
VOF_HD f2x2 two_sum(v2 a, v2 b) {
  const v2 s = vadd(a, b), bb = vsub(s, a);
  return {s, vadd(vsub(a, vsub(s, bb)), vsub(b, bb))};
}
VOF_HD f2x2 fast_two_sum(v2 a, v2 b) {
  const v2 s = vadd(a, b);
  return {s, vsub(b, vsub(s, a))};
}
VOF_HD f2x2 add(f2x2 x, f2x2 y) {
  f2x2 s = two_sum(x.hi, y.hi);
  const f2x2 t = two_sum(x.lo, y.lo);
  s.lo = vadd(s.lo, t.hi);
  s = fast_two_sum(s.hi, s.lo);
  s.lo = vadd(s.lo, t.lo);
  return fast_two_sum(s.hi, s.lo);
}
VOF_HD f2x2 add_c(f2x2 x, f2x2 y) {
  f2x2 s = two_sum(x.hi, y.hi);
  s.lo = vadd(s.lo, vadd(x.lo, y.lo));
  return fast_two_sum(s.hi, s.lo);
}
VOF_HD f2x2 mul(f2x2 x, f2x2 y) {
  const v2 p = vmul(x.hi, y.hi);
  v2 e = vfma(x.hi, y.hi, vmul(p, vset(-1.0f, -1.0f)));
  e = vfma(x.hi, y.lo, vfma(x.lo, y.hi, e));
  return fast_two_sum(p, e);
}
VOF_HD f2x2 sqr(f2x2 x) {
  const v2 p = vmul(x.hi, x.hi), m = vmul(p, vset(-1.0f, -1.0f));
  return fast_two_sum(p, vfma(vadd(x.hi, x.hi), x.lo, vfma(x.hi, x.hi, m)));
}
// times x, y (powers of two: exact)
VOF_HD f2x2 scale(f2x2 a, float x, float y) {
  const v2 f = vset(x, y);
  return {vmul(a.hi, f), vmul(a.lo, f)};
}
VOF_HD f2x2 twice(f2x2 x) { return {vadd(x.hi, x.hi), vadd(x.lo, x.lo)}; }  // exact

}  // namespace df

// Six times the WENO5 correction to the donor value (Jiang-Shu weights, eps =
// 1e-6, linear weights 0.1, 0.6, 0.3) from the four neighbour differences in upwind order, D_0
// .. D_3 (D_1 = v0 - v_-1): T_f = v0 + correction, one FP64
// fused multiply-add; exactly 0 when all four are 0.  With the second differences d_i = D_(i+1) - D_i the three
// candidates are v0 + r_k / 6, r_0 = 3 D_1 + 2 d_0, r_1 = D_1 + 2 D_2, r_2 = 3 D_2 - d_2, a = r_0 - r_1 = 2 (d_0 -
// d_1), b = r_2 - r_1 = d_1 - d_2, and six times the correction is, with p the
// candidate of the largest weight,
//   r_p + (sum over the other two of w_k (r_k - r_p)) / (w_0 + w_1 + w_2):
// only third differences pass through the weights, and a candidate across a
// jump enters by its own small weight.  (Always around r_1, a jump next to the
// central candidate's cells had to cancel in pairs: +-6e-16 of the jump on the
// mean, where three weighted candidates lose 1e-26 and this form 7e-27; over
// smooth, random, jumping and mixed stencils its mean error is at most theirs.)
// The smoothness
// indicators' first differences are 2 D_1 + d_0, D_1 + D_2 and d_2 - 2 D_2.
// Indicators scaled by 12/13 with eps (weights unchanged), linear weights by
// 10.  The differences are scaled by a power of two 2^-k with the largest near
// 1 (k >= -20) and eps by 2^-2k, both exact, so that no pair overflows or
// underflows where it matters; the correction is scaled back exactly.
// Indicators 0 and 2 mirror each other, so their arithmetic runs side by side:
// (d_0, -d_2), (e_0, -e_2), (s_0, s_2).
VOF_HD double weno5_corr6_df(double D0, double D1, double D2, double D3) {
  using namespace df;
  const words x0 = words_of(D0), x1 = words_of(D1), x2 = words_of(D2), x3 = words_of(D3);
  // exponent of the largest |D| (from the bits)
  const uint32_t h0 = x0.hi & 0x7FFFFFFFu, h1 = x1.hi & 0x7FFFFFFFu, h2 = x2.hi & 0x7FFFFFFFu, h3 = x3.hi & 0x7FFFFFFFu;
  const uint32_t m01 = h0 > h1 ? h0 : h1, m23 = h2 > h3 ? h2 : h3, mh = m01 > m23 ? m01 : m23;
  if ((mh | x0.lo | x1.lo | x2.lo | x3.lo) == 0) return 0.0;
  int k = (int)(mh >> 20) - 1023 + 1;  // max |D| < 2^k
  if (k < -20) k = -20;
  // (the outer two negated, by their sign bits)
  const f2 n0 = split_scaled({x0.hi ^ 0x80000000u, x0.lo}, k), a1 = split_scaled(x1, k), a2 = split_scaled(x2, k),
           n3 = split_scaled({x3.hi ^ 0x80000000u, x3.lo}, k);
  // eps' = 1e-6 * 12/13 * 2^-2k, exact scaling of the FP32 pair of eps'
  const f2 eps = split_scaled(words_of(1e-6 * (12.0 / 13.0)), 2 * k);
  const f2 c3 = split_scaled(words_of(3.0 / 13.0), 0);  // the ratio of the indicators' two terms, to pair accuracy
  const f2x2 A = both(a1, a2);
  const f2x2 d02 = add(A, both(n0, n3));  // (relative accuracy: they cancel)
  const f2x2 e02 = add_c(twice(A), d02);
  const f2x2 c33 = both(c3, c3), ee = both(eps, eps);
  const f2x2 s02 = sqr(add_c(add_c(sqr(d02), mul(sqr(e02), c33)), ee));
  const f2x2 de1 = add(both(a2, a2), both(neg(a1), a1));  // d_1, e_1
  f2 q0, q1, d1, e1, s0, s2;
  each(sqr(de1), q0, q1);
  const f2 s1 = sqr(add_c(add_c(q0, mul(q1, c3)), eps));
  each(s02, s0, s2);
  each(de1, d1, e1);
  // w_0 = s1 s2, w_1 = 6 s0 s2, w_2 = 3 s0 s1
  f2 w0, w2;
  each(mul(both(s2, s0), both(s1, s1)), w0, w2);
  const f2 w1 = mul_k(mul(s0, s2), 6.0f);
  w2 = mul_k(w2, 3.0f);
  const f2 W = add_c(add_c(w0, w1), w2);
  // the candidate of the largest weight and its differences to the other two:
  // (a, b) = (r_0 - r_1, r_2 - r_1)
  f2 a, b, r0, r2;
  each(scale(add_c(d02, both(neg(d1), d1)), 2.0f, 1.0f), a, b);
  each(add_c(add_c(A, twice(A)), scale(d02, 2.0f, 1.0f)), r0, r2);  // 3 D_1 + 2 d_0, 3 D_2 - d_2
  const bool p0 = w0.hi > w1.hi && w0.hi >= w2.hi, p2 = w2.hi > w1.hi && !p0;
  const f2 c = add_c(a, neg(b));
  f2 m0, m2;
  each(mul(both(p0 ? w1 : w0, p2 ? w1 : w2), both(p0 ? neg(a) : (p2 ? c : a), p2 ? neg(b) : (p0 ? neg(c) : b))), m0, m2);
  const f2 num = add_c(m0, m2), rp = p0 ? r0 : (p2 ? r2 : add_c(twice(a2), a1));
  // num / W: the FP32 quotient and one correction from its remainder
  const float qh = num.hi / W.hi;
  const f2 p = two_prod(qh, W.hi);
  const float rem = ((num.hi - p.hi) - p.lo) + (num.lo - qh * W.lo);
  const f2 q = fast_two_sum(qh, rem / W.hi);
  return widen_pair(add(rp, q), k);
}

// Donor value plus a sixth of x, one rounding; x = 0 leaves the value's bits.
VOF_HD double weno5_add6(double v0, double x) {
#ifdef __CUDA_ARCH__
  const double t = fma(x, 1.0 / 6.0, v0);
#else
  const double t = std::fma(x, 1.0 / 6.0, v0);
#endif
  const df::words w = df::words_of(x);
  return ((w.hi & 0x7FFFFFFFu) | w.lo) == 0 ? v0 : t;
}

}  // namespace vofgb
