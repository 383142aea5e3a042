// Particles of one event in light-cone form with their angles in fixed point: what the event
// kernels (jagged.cu, select.cu) stage once per particle and read once per pair.
//
// eta and phi are staged as 64-bit integers in units of 2^-59 (|eta| < 8), rounded to nearest: an
// angle difference is then one exact integer subtraction, and its reduction to the table step
// (h = d/2 = n 2^-8 + r) is bit fields of it.  An FP64 subtraction instead holds the FP64 pipe for
// ~77 cycles per warp and is followed by a conversion of the difference by its bits; the integer
// route issues about as many instructions and leaves that pipe idle.  A difference carries about
// 2^-59 of rounding from its two angles, so S = sinh^2(d_eta/2) + sin^2(d_phi/2) keeps 2^-47
// relative where it is at least 2^-22 (kFxMinS); nearer pairs go to the elementwise arithmetic,
// which subtracts the angles in FP64.  What a small angle or difference enters by itself (a
// particle's components and their gradients, d/deta and d/dphi of a pair) is formed from the doubles
// below 2^-12 (own_reduce, event_lc_grad.cuh).
#pragma once

#include "mass_lc.cuh"

namespace gvx {
namespace ffm {

constexpr float kFxMinS = 2.384185791015625e-07f;  // 2^-22

// x, |x| < 8, in units of 2^-59, rounded to nearest (ties away from zero), a nonzero x to at least one
// unit: 0 stands for 0 alone (or |x| < 2^-1042), and the sign is kept.
GVX_HD int64_t angle_fx(double x) {
  const uint32_t wh = dhi(x), wl = dlo(x);
  // the significand with one guard bit, at the place it has for x in [4, 8)
  const uint64_t M = (((uint64_t)((wh & 0xfffffu) | 0x100000u) << 32) | wl) << 10;
  // |x| raised to 2^-60; 0 wraps around and stays
  const uint32_t h = umax32((wh & 0x7fffffffu) - 1u, (963u << 20) - 1u) + 1u;
  const uint32_t sh = 1025u - (h >> 20);
  const uint64_t v = sh < 64u ? M >> sh : 0;
  const int64_t r = (int64_t)((v + 1) >> 1);
  return (wh >> 31) ? -r : r;
}

// |d|/2 = n 2^-8 + r for a difference d of two angles (units 2^-59): n to nearest, r exact to
// 2^-58 of the largest r (an integer below 2^51 in units of 2^-60 in two floats: its leading
// bits rounded by one conversion, the rest by another).
GVX_HD ff fx_half_reduce(int64_t d, uint32_t *n) {
  const int32_t dh = (int32_t)(d >> 32);
  const uint32_t dl = (uint32_t)d;
  const int32_t k = ((dh >> 19) + 1) >> 1;  // (d + 2^51) >> 52
  const int32_t rh = (int32_t)((uint32_t)dh - ((uint32_t)k << 20));
  const int32_t t = (int32_t)(((uint32_t)rh << 11) | (dl >> 21));  // r >> 21, |t| <= 2^30
  const float hi = i2f(t);
#if defined(__CUDA_ARCH__)
  const int32_t th = __float2int_rn(hi);
#else
  const int32_t th = (int32_t)hi;
#endif
  const float lo = i2f((int32_t)(((uint32_t)(t - th) << 21) + (dl & 0x1fffffu)));
  *n = (uint32_t)(k < 0 ? -k : k);
  // 2^-39 and 2^-60, negated for a negative difference
  const uint32_t sg = (uint32_t)dh & 0x80000000u;
  return {fmul(hi, u2f((88u << 23) | sg)), fmul(lo, u2f((67u << 23) | sg))};
}

// Whether an angle or a difference of two (units 2^-59) is nearer than 2^-12 to 0, where the rounding
// to units is more than 2^-48 of it.
GVX_HD uint32_t fx_near0(int64_t d) { return (uint32_t)((int32_t)(d >> 32) + (1 << 15)); }
GVX_HD bool fx_small(int64_t d) { return fx_near0(d) < (1u << 16); }
GVX_HD bool fx_small(int64_t d, int64_t e) { return umin32(fx_near0(d), fx_near0(e)) < (1u << 16); }  // either

// |x| = n 2^-8 + r of a particle's own angle x, staged as a: fx_half_reduce of 2 a, for a small angle
// r from x itself.  sinh(eta) and sin(phi) are factors of the particle's components, which keep
// their relative accuracy however small the angle.
GVX_HD ff own_reduce(double x, int64_t a, uint32_t *n) {
  ff r = fx_half_reduce(2 * a, n);
  if (fx_small(a)) r = cvt1(cvt_parts(dhi(x) & 0x7fffffffu, dlo(x), kRebaseOne));  // n is 0
  return r;
}

// d_phi modulo 2 pi into about [-pi, pi] (2 pi to 2^-60: the difference stays good to 2^-59 where
// the elementwise arithmetic has to leave |d_phi| near 2 pi to its FP64 formulas; sin^2 does not
// see the turn).
constexpr int64_t kTwoPiFx = 0x3243f6a8885a308dll;  // 2 pi in units of 2^-59
GVX_HD int64_t wrap_fx(int64_t d) {
  const int32_t dh = (int32_t)(d >> 32), half = (int32_t)(kTwoPiFx >> 33);
  if (dh > half) d -= kTwoPiFx;
  if (dh < -half) d += kTwoPiFx;
  return d;
}

// The angular factor S of a pair from its staged angles; false where it is below kFxMinS (the caller
// takes the elementwise arithmetic).
GVX_HD bool lc_pair_S_fx(int64_t eta1, int64_t phi1, int64_t eta2, int64_t phi2, const LcTab &T,
                         ff *S) {
  uint32_t n, j;
  const ff re = fx_half_reduce(eta1 - eta2, &n), rp = fx_half_reduce(wrap_fx(phi1 - phi2), &j);
  const gvx_f4 th = ldtab(&T.hyp[umin32(n, GVX_HYP_N)]);
  const gvx_f4 ts = ldtab(&T.sin[umin32(j, GVX_SIN_N)]);
  const ff2 A = {mk2(th.z, ts.x), mk2(th.w, ts.y)};
  const ff2 B = {mk2(th.x, ts.z), mk2(th.y, ts.w)};
  const ff2 w = lc_sqr(tab_eval(A, B, pack(re, rp), mk2(0.5f, -0.5f)));
  *S = lc_add(lane_x(w), lane_y(w));
  return S->hi >= kFxMinS;
}

// Whether a particle (its high words: pt with sign, |m|, |eta|, |phi|) lies in the float-float
// domain of mass_lc.cuh at its event's scale word wmax.
GVX_HD bool lc_in_domain(uint32_t hp, uint32_t hm, uint32_t he, uint32_t hf, uint32_t wmax) {
  return wmax - (200u << 20) < (1700u << 20) &&
         umin32(hp - 0x100000u, hm - 0x100000u) >= (wmax & 0x7ff00000u) - (41u << 20) &&
         umax32(hp, hm) >= 0x100000u && he < 0x40200000u && hf < 0x400C0000u;
}

// One staged particle.
struct alignas(16) EvPart {
  gvx_f4 dy;         // (D.hi, Y.hi, D.lo, Y.lo): D and Y of a pair's legs add as lanes
  int64_t eta, phi;  // units of 2^-59
  float pt_hi, pt_lo;
  uint32_t scale;    // the event's scale field; 0: outside the float-float domain, nothing else is set
  uint32_t tag;      // the caller's
};

// The scaled m^2 of a pair from its staged particles (both on the fast path, of one event); false
// where the caller has to take the elementwise arithmetic (S below kFxMinS, or m^2 nonzero and below
// 2^-80).
GVX_HD bool ev_pair_m2(const EvPart &a, const EvPart &b, const LcTab &T, ff *m2s) {
  ff S;
  const bool ok = lc_pair_S_fx(a.eta, a.phi, b.eta, b.phi, T, &S);
  const ff2 s = lc_add(ff2{mk2(a.dy.x, a.dy.y), mk2(a.dy.z, a.dy.w)},
                       ff2{mk2(b.dy.x, b.dy.y), mk2(b.dy.z, b.dy.w)});
  const ff ta = lc_mul(lc_mul(ff{a.pt_hi, a.pt_lo}, ff{b.pt_hi, b.pt_lo}), S);
  *m2s = lc_add(lc_mul(lane_x(s), lane_y(s)), ff{fmul(ta.hi, 4.0f), fmul(ta.lo, 4.0f)});
  return ok && (m2s->hi >= 8.27180613e-25f || m2s->hi == 0.0f);  // 2^-80
}

// Whether a staged angle is the FP64 one exactly: its last bit is at least 2^-59 from 2^-7 on.
GVX_HD bool fx_exact(int64_t a) { return (a < 0 ? -a : a) > (1ll << 52) || a == 0; }


// Whether both angles of a staged particle are exact, from them or from the high words of |eta| and |phi|
// (0 wraps around).
GVX_HD bool ev_exact(int64_t eta, int64_t phi) { return fx_exact(eta) && fx_exact(phi); }
GVX_HD bool ev_exact(uint32_t he, uint32_t hf) { return umin32(he - 1u, hf - 1u) >= (1016u << 20) - 1u; }

}  // namespace ffm
}  // namespace gvx
