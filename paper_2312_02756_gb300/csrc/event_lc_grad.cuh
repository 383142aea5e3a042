// The adjoint of one pair mass from two staged particles of an event (event_lc.cuh), in the form
// that the jagged adjoint (jagged_bwd.cu) sums: five numbers per pair, each of which enters both
// legs' gradients with the same or the opposite sign, so that a particle's gradient is a signed sum
// over its pairs and reads nothing of its partners.
//
// With F = m^2 = (D_a + D_b)(Y_a + Y_b) + 4 pt_a pt_b S (mass_lc_grad.cuh) and c = gm / (2 m):
//   W  = c (Y_a D_b - D_a Y_b)          + for a, - for b
//   Z  = 2 c (E_a + E_b)                + for both
//   U  = 4 c pt_a pt_b S                + for both
//   Ve = 2 c pt_a pt_b sinh(eta_a - eta_b),   Vp = 2 c pt_a pt_b sin(phi_a - phi_b)    + for a, - for b
// and with the sums of them over particle i's pairs, signed for i,
//   d/dpt_i  = (cosh eta_i / E_i) W + U / pt_i,     d/deta_i = (pt_i sinh eta_i / E_i) W + Ve,
//   d/dphi_i = Vp,                                   d/dm_i   = (m_i / E_i) Z.
// The five are carried times 2^32, so that the smallest of them stay inside the float range.
#pragma once

#include "event_lc.cuh"
#include "mass_lc_grad.cuh"

namespace gvx {
namespace ffm {

constexpr uint32_t kGradShift = 32u << 20;  // the factor 2^32, in a double's exponent field

struct EvGrad {
  ff2 we, zu;  // lanes (W, Ve) and (Z, U)
  ff vp;
};

// |d|/2 of a small difference as ff (the table step is 0).
GVX_HD ff small_half(double d) { return cvt1(cvt_parts(dhi(d) & 0x7fffffffu, dlo(d), kRebaseHalf)); }

// The angular terms from staged angles: S = sinh^2(d_eta/2) + sin^2(d_phi/2) and
// sd = (2 sinh d_eta, 2 sin d_phi), each of which enters a component of the gradient by itself, so that
// either difference has to be good relatively.  It is where it is at least 2^-12 (to 2^-47) or between
// exact angles (exact: all four are); of the others, about one pair in 10^6, near(d) gives the FP64
// differences d[0], d[1] of the angles themselves.  False where it cannot, or where S is below kFxMinS
// after a turn taken off d_phi.  (A turned d_phi is good to 2^-60, better than the FP64 difference.)
template <class Near>
GVX_HD bool lc_pair_angles_fx(int64_t eta1, int64_t phi1, int64_t eta2, int64_t phi2, bool exact, const Near &near,
                              const LcTab &T, ff *S, ff2 *sd) {
  uint32_t n, j;
  const int64_t de = eta1 - eta2, raw = phi1 - phi2, dp = wrap_fx(raw);
  ff re = fx_half_reduce(de, &n), rp = fx_half_reduce(dp, &j);
  uint32_t se = (uint32_t)(de >> 32), sp = (uint32_t)(dp >> 32);
  bool good = true;
  if (__builtin_expect((int)fx_small(de, dp) & (int)!exact, 0)) {
    double d[2] = {0.0, 0.0};
    good = near(d);
    if (fx_small(de)) {
      re = small_half(d[0]);
      se = dhi(d[0]);
    }
    if (fx_small(dp) && dp == raw) {
      rp = small_half(d[1]);
      sp = dhi(d[1]);
    }
  }
  const gvx_f4 th = ldtab(&T.hyp[umin32(n, GVX_HYP_N)]);
  const gvx_f4 ts = ldtab(&T.sin[umin32(j, GVX_SIN_N)]);
  const ff2 A = {mk2(th.z, ts.x), mk2(th.w, ts.y)};     // (sinh, sin) of the table point
  const ff2 B = {mk2(th.x, ts.z), mk2(th.y, ts.w)};     // (cosh, cos)
  const ff2 Bn = {mk2(th.z, -ts.x), mk2(th.w, -ts.y)};  // (sinh, -sin)
  // the leading parts are in steps of 2^-39 and |hi| >= |lo| or hi = 0: normalised for the small ones
  const ff2 r = fast_two_sum2(mk2(re.hi, rp.hi), mk2(re.lo, rp.lo));
  const TabPoly<f2> tp = tab_poly(r, mk2(0.5f, -0.5f));
  const ff2 w = tab_comb(A, B, r, tp), wc = tab_comb_any(B, Bn, r, tp);
  const ff2 w2 = lc_sqr(w);
  *S = lc_add(lane_x(w2), lane_y(w2));
  *sd = lc_scale(lc_mul(w, wc), mk2(u2f(0x40800000u | (se & 0x80000000u)), u2f(0x40800000u | (sp & 0x80000000u))));  // +-4
  return good && (S->hi >= kFxMinS || dp == raw);
}

// |gm| in [2^-60, 2^20], or gm = 0.
GVX_HD bool ev_grad_in_range(double g) {
  const uint32_t hg = dhi(g) & 0x7fffffffu;
  return hg - (963u << 20) < (81u << 20) || (hg | dlo(g)) == 0u;
}

// The five terms of a pair, times 2^32 (exact, near: lc_pair_angles_fx); false where the caller has to
// take the elementwise formulas (angles that the staged ones do not give, m^2 nonzero and below 2^-80,
// gm out of range).
template <class Near>
GVX_HD bool ev_pair_grad(const EvPart &a, const EvPart &b, bool exact, const Near &near, double g, const LcTab &T,
                         EvGrad *o) {
  ff S;
  ff2 sd;
  const bool ok = lc_pair_angles_fx(a.eta, a.phi, b.eta, b.phi, exact, near, T, &S, &sd);
  const ff2 s = lc_add(ff2{mk2(a.dy.x, a.dy.y), mk2(a.dy.z, a.dy.w)},
                       ff2{mk2(b.dy.x, b.dy.y), mk2(b.dy.z, b.dy.w)});  // (D_a + D_b, Y_a + Y_b)
  const ff p12 = lc_mul(ff{a.pt_hi, a.pt_lo}, ff{b.pt_hi, b.pt_lo});
  const ff ta = lc_scale(lc_mul(p12, S), 4.0f);
  const ff m2s = lc_add(lc_mul(lane_x(s), lane_y(s)), ta);
  const uint32_t hg = dhi(g) & 0x7fffffffu;
  if (m2s.hi == 0.0f || (hg | dlo(g)) == 0u) {  // m = 0 or gm = 0: no contribution
    *o = EvGrad{{bc2(0.0f), bc2(0.0f)}, {bc2(0.0f), bc2(0.0f)}, {0.0f, 0.0f}};
    return ok && (S.hi == 0.0f || (hg | dlo(g)) == 0u);  // m^2 below the floats is not 0
  }
  const ff m = lc_sqrt_refined(m2s);
  const ff gf = cvt1(cvt_parts(hg, dlo(g), kRebaseOne - kGradShift));
  const ff c = lc_scale(lc_div(gf, m), 0.5f * sign_of(g));
  const ff2 yd = lc_mul(ff2{mk2(a.dy.y, a.dy.x), mk2(a.dy.w, a.dy.z)},
                        ff2{mk2(b.dy.x, b.dy.y), mk2(b.dy.z, b.dy.w)});  // (Y_a D_b, D_a Y_b)
  const ff N = lc_sum(lane_x(yd), lc_scale(lane_y(yd), -1.0f));
  const ff E2 = lc_add(lane_x(s), lane_y(s));  // 2 (E_a + E_b)
  const ff2 cb = {bc2(c.hi), bc2(c.lo)};
  const ff cp = lc_mul(c, p12);
  const ff2 v = lc_mul(ff2{bc2(cp.hi), bc2(cp.lo)}, sd);
  const ff W = lc_mul(c, N);
  o->we = pack(W, lane_x(v));
  o->zu = lc_mul(cb, pack(E2, ta));
  o->vp = lane_y(v);
  return ok && m2s.hi >= 8.27180613e-25f && ev_grad_in_range(g);  // 2^-80
}
// The same from the staged particles alone.
GVX_HD bool ev_pair_grad(const EvPart &a, const EvPart &b, double g, const LcTab &T, EvGrad *o) {
  return ev_pair_grad(a, b, ev_exact(a.eta, a.phi) && ev_exact(b.eta, b.phi), [](double *) { return false; }, g, T, o);
}

// ---- a particle's own part --------------------------------------------------------------------
// Lane-generic (mass_lc.cuh): F = ff for one particle, ff2 for two at once as the lanes of paired FP32
// instructions, each at its event's scale.

// x with the sign of the double of high word w.
GVX_HD ff with_sign(const ff &x, uint32_t w) {
  const uint32_t s = w & 0x80000000u;
  return {u2f(f2u(x.hi) ^ s), u2f(f2u(x.lo) ^ s)};
}

// What is read of a particle: pt, Y, D and m at the scale, eta and phi as 2^-8 n + r (of the
// absolute value) and their signs.
template <class F>
struct EvOwn {
  F pt, Y, D, mm, re, rp;
  uint32_t n[2], j[2];
  lane_t<F> seta, sphi;
};
GVX_HD EvOwn<ff> ev_own(const EvPart &p, const ff &mm) {
  EvOwn<ff> o;
  o.pt = {p.pt_hi, p.pt_lo};
  o.Y = {p.dy.y, p.dy.w};
  o.D = {p.dy.x, p.dy.z};
  o.mm = mm;
  o.re = fx_half_reduce(2 * p.eta, &o.n[0]);
  o.rp = fx_half_reduce(2 * p.phi, &o.j[0]);
  o.n[1] = o.j[1] = 0u;
  o.seta = p.eta < 0 ? -1.0f : 1.0f;
  o.sphi = p.phi < 0 ? -1.0f : 1.0f;
  return o;
}
GVX_HD EvOwn<ff2> pack(const EvOwn<ff> &a, const EvOwn<ff> &b) {
  return {pack(a.pt, b.pt), pack(a.Y, b.Y),   pack(a.D, b.D),       pack(a.mm, b.mm),
          pack(a.re, b.re), pack(a.rp, b.rp), {a.n[0], b.n[0]},     {a.j[0], b.j[0]},
          mk2(a.seta, b.seta), mk2(a.sphi, b.sphi)};
}

// 1/E, cosh(eta), m/E and pt sinh(eta), sinh(eta) (signed).
template <class F>
struct EvLeg {
  F rE, ch, sh, psh, mE;
};
template <class F>
GVX_HD EvLeg<F> ev_leg(const EvOwn<F> &o, const LcTab &T) {
  using V = lane_t<F>;
  EvLeg<F> l;
  F C, Sh;
  tab_load(T.hyp, GVX_HYP_N, o.n, &C, &Sh);
  const TabPoly<V> tp = tab_poly(o.re, vbc(0.5f, V{}));
  l.ch = tab_comb(C, Sh, o.re, tp);
  l.sh = lc_scale(tab_comb(Sh, C, o.re, tp), o.seta);
  const F E2 = lc_add(o.Y, o.D);  // 2 E
  l.rE = lc_div(F{vbc(2.0f, V{}), vbc(0.0f, V{})}, E2);
  l.psh = lc_mul(o.pt, l.sh);
  l.mE = lc_mul(o.mm, l.rE);
  return l;
}

// The pair part of the gradient from the sums over the particle's pairs.
template <class F>
GVX_HD void ev_grad_terms(const EvOwn<F> &o, const EvLeg<F> &l, const F &W, const F &Ve, const F &Z,
                          const F &U, F *dpt, F *deta, F *dm) {
  const F w = lc_mul(W, l.rE);
  *dpt = lc_sum(lc_mul(l.ch, w), lc_div(U, o.pt));
  *deta = lc_sum(lc_mul(l.psh, w), Ve);
  *dm = lc_mul(l.mE, Z);
}

// J^T gs, J = d(px, py, pz, E)/d(pt, eta, phi, m) of the particle.
template <class F>
GVX_HD void ev_sum_terms(const EvOwn<F> &o, const EvLeg<F> &l, const F *gs, const LcTab &T, F *t) {
  using V = lane_t<F>;
  F Sj, Cj;
  tab_load(T.sin, GVX_SIN_N, o.j, &Sj, &Cj);
  const TabPoly<V> tp = tab_poly(o.rp, vbc(-0.5f, V{}));
  const F sn = lc_scale(tab_comb_any(Sj, Cj, o.rp, tp), o.sphi);
  const F cs = tab_comb_any(Cj, F{vneg(Sj.hi), vneg(Sj.lo)}, o.rp, tp);
  const F P = lc_mul(o.pt, l.ch);
  const F gEP = lc_mul(lc_mul(gs[3], l.rE), P);
  const F gxs = lc_mul(gs[0], sn);
  t[0] = lc_sum(lc_sum(lc_mul(gs[0], cs), lc_mul(gs[1], sn)), lc_sum(lc_mul(gs[2], l.sh), lc_mul(gEP, l.ch)));
  t[1] = lc_sum(lc_mul(gs[2], P), lc_mul(gEP, l.psh));
  t[2] = lc_mul(o.pt, lc_sum(lc_mul(gs[1], cs), F{vneg(gxs.hi), vneg(gxs.lo)}));
  t[3] = lc_mul(gs[3], l.mE);
}

// gs at its own scale 2^sg: its scale field, 0 when it is zero, or 1 when a component lies outside
// [2^-300, 2^300] (the caller takes the FP64 formulas).
GVX_HD uint32_t ev_gs(double g0, double g1, double g2, double g3, ff *g) {
  const double v[4] = {g0, g1, g2, g3};
  uint32_t hmax = 0, low = 0;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    hmax = umax32(hmax, dhi(v[k]) & 0x7fffffffu);
    low |= dlo(v[k]);
  }
  const bool zero = (hmax | low) == 0u, ok = hmax - (723u << 20) < (600u << 20);
  const uint32_t ew = ok ? hmax & 0x7ff00000u : 1023u << 20, rb = ew - (127u << 20);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    g[k] = with_sign(cvt1(cvt_parts(dhi(v[k]) & 0x7fffffffu, dlo(v[k]), rb)), dhi(v[k]));
  }
  return zero ? 0u : ok ? ew : 1u;
}

// ff times 2^shift -> double (eoff = (896 + shift) << 20), for any ratio of hi and lo.
GVX_HD double ev_out(const ff &x, uint32_t eoff) { return lc_to_double_int(two_sum(x.hi, x.lo), eoff); }

// The exponent offsets of the outputs at the event's scale field ew: of the pair part (its sums carry
// 2^32), d/dpt and d/dm first, d/deta and d/dphi second; and of the event-sum part at gs's field ewg.
GVX_HD uint32_t ev_off_pt() { return (896u << 20) - kGradShift; }
GVX_HD uint32_t ev_off_angle(uint32_t ew) { return ew - (127u << 20) - kGradShift; }
GVX_HD uint32_t ev_off_gs_pt(uint32_t ewg) { return ewg - (127u << 20); }
GVX_HD uint32_t ev_off_gs_angle(uint32_t ewg, uint32_t ew) { return ewg + ew - (1150u << 20); }

}  // namespace ffm
}  // namespace gvx
