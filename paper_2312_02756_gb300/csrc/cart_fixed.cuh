// Pair mass of PxPyPzE legs in exact fixed-point integer arithmetic: the fast path of the
// Cartesian-input mass kernels (the mass kernel of Sec. 4.1 on the PxPyPzE system of Sec. 3.1).
//
// The plain definition m^2 = (E1 + E2)^2 - (px1 + px2)^2 - (py1 + py2)^2 - (pz1 + pz2)^2 cancels
// catastrophically in floating point for light, collinear pairs.  Here the eight components are
// scaled by the power of two 2^-sc that brings the largest magnitude into [1, 2) and truncated to
// integers in units of 2^-83 (magnitudes below 2^84), held as three signed limbs of 28 bits.  The
// component sums are then exact limb by limb, with no carry to pass on, and a sum's square is five
// 32 x 32 -> 64-bit multiply-adds, collected over the components by weight in four 64-bit sums that
// are put together once.  The only errors are the truncations: in scaled units |error of m^2| <
// 4 (2 * 4 * 2^-82) + 2^-100 < 2^-76.9.  The result is kept when |m^2| >= 2^-31 (scaled), i.e. with
// relative error below 2^-45.9; it is then rounded to float-float (47 bits), its square root
// taken in float-float, and scaled back: the relative error of m is below 2^-44.  Integer and FP32
// pipes only, plus one FP64 add for the final rounding (none for FP32 output).
//
// Bound by issue with the loads (10,000,019 FP64 pairs as rows: 143 us, 5.0 TB/s of the 72 bytes a pair,
// 420 warp instructions per 32 pairs).  In the same launch shape (256 threads) it took 153 us, and three
// 32-bit words per magnitude, with compares for the signs of the sums and carries through every product,
// 188 us and 511 instructions.
//
// Outside the fast path (a non-finite component, a scale exponent outside [-900, 900] for double
// or [-100, 100] for float input, a denormal float at a scale exponent below -43, or |m^2| below the
// threshold, zero included) the functions return false and the caller evaluates the cancellation-free
// FP64 form.
#pragma once

#include "ff.cuh"
#include "mass_ff2.cuh"

namespace gvx {
namespace cfix {

using ffm::ff;
typedef unsigned __int128 u128;
typedef __int128 i128;

constexpr int kFrac = 83;                 // input units: 2^-83 of the scale
constexpr int kM2Units = 2 * kFrac - 64;   // m^2 units: 2^-102
constexpr int kMinLead = kM2Units - 31;    // |m^2| >= 2^-31: leading bit at or above 71
constexpr int kLimb = 28;                  // bits of a limb: three hold a magnitude below 2^84
constexpr uint32_t kLimbMask = (1u << kLimb) - 1;

// 32-bit shifts by n >= 0 that give 0 (the upper word, for a funnel) at and beyond 32.
GVX_HD uint32_t shr_c(uint32_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_rc(x, 0u, n);
#else
  return n < 32u ? x >> n : 0u;
#endif
}
GVX_HD uint32_t shl_c(uint32_t x, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_lc(0u, x, n);
#else
  return n < 32u ? x << n : 0u;
#endif
}
GVX_HD uint32_t funnel_rc(uint32_t lo, uint32_t hi, uint32_t n) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_rc(lo, hi, n);
#else
  return n < 32u ? (uint32_t)((((uint64_t)hi << 32) | lo) >> n) : hi;
#endif
}

// a b + c, 32 x 32 -> 64 bits signed.
GVX_HD int64_t mad_wide(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }

// Format constants: kBias, kMaxE (the Inf/NaN exponent), kScaleLim (allowed |scale exponent|), kExpBit
// (the exponent's lowest bit in the upper word).
template <typename T>
struct Fmt;
template <>
struct Fmt<double> {
  static constexpr int kBias = 1023, kMaxE = 0x7ff, kScaleLim = 900, kExpBit = 20;
};
template <>
struct Fmt<float> {
  static constexpr int kBias = 127, kMaxE = 0xff, kScaleLim = 100, kExpBit = 23;
};

GVX_HD uint32_t top_word(double x) { return ffm::dhi(x); }
GVX_HD uint32_t top_word(float x) { return ffm::f2u(x); }

// The significand with its leading bit at bit 63, as two words.  A zero or denormal counts as 0 (it
// lies below the units; m2_fixed declines the lowest FP32 scales, where a denormal does not): a float's
// significand is cleared here, because at scale exponent -100 its exponent field of 0 is only 27
// binades down; a double's, at least 123 binades down, is shifted out of the outer limbs by limbs_near,
// which masks the middle one.
struct Sig {
  uint32_t hi, lo;
};
GVX_HD Sig significand(double x, uint32_t wh) {
  const uint32_t h = (wh & 0xfffffu) | 0x100000u, l = ffm::dlo(x);
  return {(h << 11) | (l >> 21), l << 11};
}
GVX_HD Sig significand(float, uint32_t w) { return {(w & 0x7f800000u) ? (w << 8) | 0x80000000u : 0u, 0u}; }

// A value of the scaled fixed point, in limbs of kLimb bits (those of a sum of two may be
// negative or one bit longer).
struct Limbs {
  int32_t s0, s1, s2;
};
// |x| 2^(kFrac - sc) truncated, d binades below the scale: the significand at the top of the 84 bits,
// moved right by d <= 20 (a shift per limb) ...
GVX_HD Limbs limbs_near(const Sig &t, uint32_t d, bool zero) {
  return {(int32_t)(shl_c(t.lo, 20u - d) & kLimbMask),
          (int32_t)(funnel_rc(t.lo, t.hi, 8u + d) & (zero ? 0u : kLimbMask)),
          (int32_t)shr_c(t.hi, 4u + d)};
}
// ... or by any d (components more than 20 binades apart).
GVX_HD Limbs limbs_far(const Sig &t, uint32_t d, bool zero) {
  if (d <= 20u || zero) return limbs_near(t, d, zero);
  const uint64_t T = ((uint64_t)t.hi << 32) | t.lo, v = d < 84u ? T >> (d - 20u) : 0;
  return {(int32_t)((uint32_t)v & kLimbMask), (int32_t)((uint32_t)(v >> kLimb) & kLimbMask),
          (int32_t)(uint32_t)(v >> (2 * kLimb))};
}

// The scaled m^2 (units 2^-102) of two PxPyPzE legs and the scale exponent sc; false when a
// component is not finite or sc is out of range.
template <typename T>
GVX_HD bool m2_fixed(const T *a, const T *b, i128 *m2, int *sc) {
  constexpr int kB = Fmt<T>::kExpBit;
  uint32_t w[8], wmax = 0, wmin = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    w[k] = top_word(k < 4 ? a[k & 3] : b[k & 3]);
    const uint32_t m = w[k] & 0x7fffffffu;
    wmax = m > wmax ? m : wmax;
    const uint32_t z = m - (1u << kB);  // zeros and denormals wrap around: they do not count
    wmin = z < wmin ? z : wmin;
  }
  const int emax = (int)(wmax >> kB), s = emax - Fmt<T>::kBias;
  if (emax == Fmt<T>::kMaxE || s < -Fmt<T>::kScaleLim || s > Fmt<T>::kScaleLim) return false;
  if constexpr (sizeof(T) == 4) {  // a denormal component (below 2^-126) above the units of the scale
    if (s < kFrac - 126) {
#pragma unroll
      for (int k = 0; k < 8; k++)
        if ((w[k] & 0x7fffffffu) - 1u < 0x7fffffu) return false;
    }
  }
  const bool far = (uint32_t)emax - ((wmin + (1u << kB)) >> kB) > 20u;
  // the sums of the components, limb by limb and without carries
  Limbs S[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    Limbs v[2];
#pragma unroll
    for (int l = 0; l < 2; l++) {
      const uint32_t wk = w[k + 4 * l], m = wk & 0x7fffffffu;
      const bool zero = m < (1u << kB);
      const Sig t = significand(l ? b[k] : a[k], wk);
      const uint32_t d = (uint32_t)emax - (m >> kB);
      const int32_t sg = ((int32_t)wk >> 31) | 1;
      const Limbs u = far ? limbs_far(t, d, zero) : limbs_near(t, d, zero);
      v[l] = {u.s0 * sg, u.s1 * sg, u.s2 * sg};
    }
    S[k] = {v[0].s0 + v[1].s0, v[0].s1 + v[1].s1, v[0].s2 + v[1].s2};
  }
  // their squares by weight: limbs below 2^29, so three of them and the cross terms stay inside 63
  // bits; s0^2 is below the resolution
  int64_t p[4] = {0, 0, 0, 0}, e[4] = {0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const Limbs &v = S[k];
    const int32_t t1 = 2 * v.s1, t0 = 2 * v.s0;
    int64_t *c = k == 3 ? e : p;  // components 0..2 are p, 3 is E
    c[3] = mad_wide(v.s2, v.s2, c[3]);
    c[2] = mad_wide(v.s2, t1, c[2]);
    c[1] = mad_wide(v.s1, v.s1, mad_wide(v.s2, t0, c[1]));
    c[0] = mad_wide(v.s1, t0, c[0]);
  }
  *m2 = ((i128)(e[3] - p[3]) << (4 * kLimb - 64)) + ((i128)(e[2] - p[2]) << (3 * kLimb - 64)) +
        ((e[1] - p[1]) >> (64 - 2 * kLimb)) + ((e[0] - p[0]) >> (64 - kLimb));
  *sc = s;
  return true;
}

// sqrt(|m^2|) in ff (scaled) with the sign of m^2; false below the threshold.
GVX_HD bool mass_scaled(i128 m2, ff *m, bool *neg) {
  *neg = m2 < 0;
  const u128 q = *neg ? (u128)(-m2) : (u128)m2;
  const uint64_t top = (uint64_t)(q >> 64);
  if (top < ((uint64_t)1 << (kMinLead - 64))) return false;
  // the 64 bits from the leading one on: hi its 24, lo the next 23
  uint32_t h = (uint32_t)(top >> 32), g = (uint32_t)top, f = (uint32_t)((uint64_t)q >> 32);
  const bool low = h == 0u;
  if (low) {
    h = g;
    g = f;
    f = (uint32_t)q;
  }
#if defined(__CUDA_ARCH__)
  const int n = __clz((int)h);
#else
  const int n = __builtin_clz(h);
#endif
  const uint32_t x = n ? (h << n) | (g >> (32 - n)) : h, y = n ? (g << n) | (f >> (32 - n)) : g;
  const uint32_t eh = (uint32_t)((low ? 95 : 127) - n - kM2Units + 127);  // biased exponent of hi
  const uint32_t base = (eh - 23u) << 23;
  const float hi = ffm::u2f((eh << 23) | ((x >> 8) & 0x7fffffu));
  const float lo = ffm::fsub(ffm::u2f(base | (((x << 15) | (y >> 17)) & 0x7fffffu)), ffm::u2f(base));
  *m = ffm::sqrt(ff{hi, lo});
  return true;
}

// Pair mass of two FP64 PxPyPzE legs (m = -sqrt(-m^2) for a spacelike sum); false outside the
// fast path.
GVX_HD bool mass_pxpypze(const double *a, const double *b, double *out) {
  i128 m2;
  int sc;
  ff m;
  bool neg;
  if (!m2_fixed<double>(a, b, &m2, &sc) || !mass_scaled(m2, &m, &neg)) return false;
  const double r = ffm::to_double(m, sc);
  *out = neg ? -r : r;
  return true;
}

// The same for FP32 legs, rounded once to float (hi + lo in one float add, then an exact
// power-of-two scaling: the scaled mass lies in [2^-16, 2^3) and |sc| <= 100).
GVX_HD bool mass_pxpypze(const float *a, const float *b, float *out) {
  i128 m2;
  int sc;
  ff m;
  bool neg;
  if (!m2_fixed<float>(a, b, &m2, &sc) || !mass_scaled(m2, &m, &neg)) return false;
  const float r = ffm::fmul(ffm::fadd(m.hi, m.lo), ffm::pow2f(sc));
  *out = neg ? -r : r;
  return true;
}

}  // namespace cfix
}  // namespace gvx

#include "cart_pxpypzm.cuh"
