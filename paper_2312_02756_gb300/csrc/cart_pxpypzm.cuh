// Pair mass of PxPyPzM legs in float-float (the mass kernel of Sec. 4.1 on the PxPyPzM system of
// Sec. 3.1).
//
// With the mass stored, E_i = sqrt(P_i + m_i^2), P_i = |p_i|^2, is not a stored number, and
//   m^2 = m1^2 + m2^2 + 2 (E1 E2 - d),   d = p1.p2,
//   E1 E2 - d = N / (E1 E2 + d)   (d > 0),   N = E1^2 E2^2 - d^2 = |p1 x p2|^2 + P1 q2 + q1 E2^2,
//             = E1 E2 + |d|       (otherwise),   q_i = m_i^2.
// The one cancelling quantity is |p1 x p2|^2.  It does not change when a multiple of p1 is taken
// from p2: with l = d / P1 to single precision and u = p2 - l p1,
//   |p1 x p2|^2 = |p1 x u|^2 = P1 R - r^2,   R = |u|^2,   r = p1.u,
// and |u| <= (theta + 2^-22) |p2| for legs theta apart, so float-float sums of relative error
// 2^-46 leave an absolute error of 2^-46 max(theta^2, 2^-44) P1 P2: relative 2^-46 where the angle
// matters, and far below m^2's own terms where it does not.  u is one FP64 FMA per component (its
// rounding is relative to u; l has 24 bits, so the product is exact there): the only FP64 operations besides
// the final addition.  The rest of p2 enters through u as well: d = l P1 + r and
// P2 = R + l (d + r), so p2 itself is never converted.
//
// Each leg has its own power-of-two scale 2^s_i: an absolute error in m_i^2 reaches m^2
// multiplied by about E_o / E_i, so the resolution must follow each leg.  The result is kept when
// m^2 >= 2^-31 H, H the larger leg's squared scale; its relative error is below 2^-43 there.
// Domain: both legs finite with scale exponents within half the format's limit and at most 60
// apart.  Components below 2^-70 of their leg's scale count as about that (FP64; FP32 keeps them).
//
// Bound by issue (560 warp instructions per 32 pairs, 83% of the slots).  10,000,019 FP64 pairs, SoA:
// 167 us (4.3 TB/s of the 72 bytes a pair; 177 us in CTAs of 256 threads), against 385 us for the components of p1 x p2 from six exact 85-bit limb products and both legs converted
// (1,150 warp instructions per 32 pairs); the largest error against binary128 fell from 2^-44.7 to
// 2^-45.4.
#pragma once

#include "cart_fixed.cuh"
#include "mass_lc.cuh"

namespace gvx {
namespace cfix {

using ffm::ff2;

// x 2^-s as ff: hi the value rounded to 24 bits, lo the exact rest rounded to 24 bits; rb = R(e) of the
// leg's scale exponent (mass_lc.cuh).  |x| 2^-s < 2; a value below 2^-70 becomes one of about 2^-70.
GVX_HD ff scaled_ff(double x, uint32_t rb) {
  const uint32_t wh = ffm::dhi(x), wl = ffm::dlo(x), sign = wh & 0x80000000u;
  const int32_t a = (int32_t)((wh & 0x7fffffffu) - rb), low = 57 << 20;
  const uint32_t w = (uint32_t)(a > low ? a : low);
  const uint32_t rl = wl + 0x10000000u;  // rounds at hi's last bit; a carry moves into w
  const uint32_t hb = ffm::funnel_l3(rl, w + (rl < wl ? 1u : 0u)) | sign;
  const uint32_t e = (((w & 0x0ff00000u) << 3) - (55u << 23)) | sign;
  return {ffm::u2f(hb), ffm::fmul(ffm::i2f((int32_t)(wl << 3)), ffm::u2f(e))};
}
GVX_HD ff scaled_ff(float x, float k) { return {ffm::fmul(x, k), 0.0f}; }

// The leading 24 bits of x 2^-s.
GVX_HD float scaled_hi(double x, uint32_t rb) {
  const uint32_t wh = ffm::dhi(x);
  const int32_t a = (int32_t)((wh & 0x7fffffffu) - rb);
  return ffm::u2f(ffm::funnel_l3(ffm::dlo(x), (uint32_t)(a > 0 ? a : 0)) | (wh & 0x80000000u));
}
GVX_HD float scaled_hi(float x, float k) { return ffm::fmul(x, k); }

// What scales a leg with largest biased exponent e: its rebase (double) or the factor 2^-s (float).
GVX_HD uint32_t leg_scale(int e, double) { return (uint32_t)(e - 127) << 20; }
GVX_HD float leg_scale(int e, float) { return ffm::pow2f(127 - e); }

GVX_HD int exp_field(uint32_t h, double) { return (int)(h >> 20); }
GVX_HD int exp_field(uint32_t h, float) { return (int)(h >> 23); }
GVX_HD uint32_t abs_word(double x) { return ffm::dhi(x) & 0x7fffffffu; }
GVX_HD uint32_t abs_word(float x) { return ffm::f2u(x) & 0x7fffffffu; }

// u = p2 - l p1 for one component, scaled by the second leg's scale: l in scaled units, ds = s2 - s1.
GVX_HD double times_pow2(float l, int ds, double) { return ffm::f2d_bits(l, ds); }
GVX_HD float times_pow2(float l, int, float) { return l; }
GVX_HD ff residual(double p1, double p2, double l, uint32_t rb2, uint32_t) {
  return scaled_ff(fma(-l, p1, p2), rb2);
}
GVX_HD ff residual(float p1, float p2, float l, float k2, float k1) {
  const ff p = ffm::two_prod(l, ffm::fmul(p1, k1));
  const ff s = ffm::two_sum(ffm::fmul(p2, k2), -p.hi);
  return ffm::renorm({s.hi, ffm::fsub(s.lo, p.lo)});
}

// a + b + c, the leading parts summed without error and the rest collected in one float.
GVX_HD ff sum3(ff a, ff b, ff c) {
  const ff s = ffm::two_sum(a.hi, b.hi), t = ffm::two_sum(s.hi, c.hi);
  return ffm::fast_two_sum(t.hi, ffm::fadd(ffm::fadd(s.lo, t.lo), ffm::fadd(ffm::fadd(a.lo, b.lo), c.lo)));
}
GVX_HD ff2 sum3(const ff2 &a, const ff2 &b, const ff2 &c) {
  using namespace ffm;
  const ff2 s = two_sum2(a.hi, b.hi), t = two_sum2(s.hi, c.hi);
  return fast_two_sum2(t.hi, add2(add2(s.lo, t.lo), add2(add2(a.lo, b.lo), c.lo)));
}

// The scaled mass sqrt(m^2 / 2^(2 e)) in ff and the exponent e of the pair mass of two PxPyPzM
// legs; false outside the fast path.
template <typename T>
GVX_HD bool mass_pxpypzm_scaled(const T *a, const T *b, ff *m, int *e_out) {
  using namespace ffm;
  const int e1 = exp_field(umax32(umax32(abs_word(a[0]), abs_word(a[1])), umax32(abs_word(a[2]), abs_word(a[3]))), T(0));
  const int e2 = exp_field(umax32(umax32(abs_word(b[0]), abs_word(b[1])), umax32(abs_word(b[2]), abs_word(b[3]))), T(0));
  const int s1 = e1 - Fmt<T>::kBias, s2 = e2 - Fmt<T>::kBias, gap = s1 > s2 ? s1 - s2 : s2 - s1;
  const int lim = Fmt<T>::kScaleLim / 2;
  if (s1 < -lim || s1 > lim || s2 < -lim || s2 > lim || gap > 60) return false;
  const auto k1 = leg_scale(e1, T(0)), k2 = leg_scale(e2, T(0));
  // l, to single precision; 0 for a first leg (nearly) at rest, whose mass dominates then
  ff p1[3];
  float d = 0.0f, n1 = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; k++) {
    p1[k] = scaled_ff(a[k], k1);
    n1 = ffma(p1[k].hi, p1[k].hi, n1);
    d = ffma(p1[k].hi, scaled_hi(b[k], k2), d);
  }
  const float l = n1 >= 8.67361738e-19f ? fmul(d, rcp_mufu(n1)) : 0.0f;  // 2^-60
  const T lt = times_pow2(l, s2 - s1, T(0));
  // lanes: (p1, u)
  ff2 x[3];
  ff xr[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const ff u = residual(a[k], b[k], lt, k2, k1);
    x[k] = pack(p1[k], u);
    xr[k] = mul(p1[k], u);
  }
  const ff2 PR = sum3(sqr(x[0]), sqr(x[1]), sqr(x[2]));  // (P1, R)
  const ff r = sum3(xr[0], xr[1], xr[2]);
  const ff P1 = lane_x(PR), R = lane_y(PR);
  const ff dot = add_same(mul_f(P1, l), r);
  const ff P2 = add_same(R, mul_f(add_same(dot, r), l));
  const ff2 qq = sqr(pack(scaled_ff(a[3], k1), scaled_ff(b[3], k2)));
  const ff q1 = lane_x(qq), q2 = lane_y(qq);
  const ff2 EE = add_same(pack(P1, P2), qq);  // (E1^2, E2^2)
  const ff E1E2 = ffm::sqrt(mul(lane_x(EE), lane_y(EE)));  // scale 2^(s1 + s2)
  const float sg = dot.hi > 0.0f ? 1.0f : -1.0f;
  ff T2 = add_same(E1E2, scale(dot, sg));
  if (dot.hi > 0.0f) {
    const ff2 AB = mul(pack(P1, q1), pack(add_same(R, q2), lane_y(EE)));  // P1 (R + q2), q1 E2^2
    const ff N = sum3(lane_x(AB), lane_y(AB), neg(sqr(r)));
    T2 = div(N, T2);
  }
  // m^2 / 2^(s1 + s2) = q1 2^(s1 - s2) + q2 2^(s2 - s1) + 2 T; an odd s1 + s2 moves one factor 2
  // inside the root
  const int odd = (s1 + s2) & 1;
  const ff m2 = sum3(scale(q1, pow2f(s1 - s2 + odd)), scale(q2, pow2f(s2 - s1 + odd)), scale(T2, odd ? 4.0f : 2.0f));
  // threshold: m^2 >= 2^-31 2^(2 max(s1, s2)), i.e. the scaled value >= 2^(|s1 - s2| - 31 + odd)
  if (!(m2.hi >= pow2f(gap - 31 + odd))) return false;
  *m = ffm::sqrt(m2);
  *e_out = (s1 + s2 - odd) / 2;
  return true;
}

GVX_HD bool mass_pxpypzm(const double *a, const double *b, double *out) {
  ff m;
  int e;
  if (!mass_pxpypzm_scaled(a, b, &m, &e)) return false;
  *out = ffm::lc_to_double(m, (uint32_t)(896 + e) << 20);
  return true;
}

GVX_HD bool mass_pxpypzm(const float *a, const float *b, float *out) {
  ff m;
  int e;
  if (!mass_pxpypzm_scaled(a, b, &m, &e)) return false;
  *out = ffm::fmul(ffm::fadd(m.hi, m.lo), ffm::pow2f(e));
  return true;
}

}  // namespace cfix
}  // namespace gvx
