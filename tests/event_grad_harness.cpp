// Host build of the jagged adjoint's pair and particle arithmetic
// (paper_2312_02756_gb300/csrc/event_lc_grad.cuh): the same source the kernel compiles, over arrays.
#include <math.h>
#include <stdint.h>

#include "../paper_2312_02756_gb300/csrc/event_lc_grad.cuh"

using namespace gvx::ffm;

static bool stage(const double *v, uint32_t wmax, const LcTab &T, EvPart *p, ff *mm) {
  const uint32_t hp = dhi(v[0]), hm = dhi(v[3]) & 0x7fffffffu;
  if (hp < 0x100000u ||
      !lc_in_domain(hp, hm, dhi(v[1]) & 0x7fffffffu, dhi(v[2]) & 0x7fffffffu, wmax)) return false;
  const uint32_t rb = (wmax & 0x7ff00000u) - (127u << 20);
  const ff pt = cvt1(cvt_parts(hp, dlo(v[0]), rb)), m = cvt1(cvt_parts(hm, dlo(v[3]), rb));
  p->eta = angle_fx(v[1]);
  p->phi = angle_fx(v[2]);
  uint32_t n;
  const ff r = fx_half_reduce(2 * p->eta, &n);
  const LcLeg<ff> L = lc_leg_at(pt, m, r, &n, T.hyp);
  p->dy = gvx_f4{L.D.hi, L.Y.hi, L.D.lo, L.Y.lo};
  p->pt_hi = pt.hi;
  p->pt_lo = pt.lo;
  *mm = with_sign(m, dhi(v[3]));
  return true;
}

static uint32_t word(const double *v) { return umax32(dhi(v[0]), dhi(v[3]) & 0x7fffffffu); }

// The gradient of one leg of a pair, as the sums of that pair alone.
static void leg_out(const EvPart &p, const ff &m, uint32_t ew, const LcTab &T, const ff2 &we, const ff2 &zu,
                    const ff &vp, double *g) {
  const EvOwn<ff> o = ev_own(p, m);
  ff dpt, deta, dm;
  ev_grad_terms(o, ev_leg(o, T), lane_x(we), lane_y(we), lane_x(zu), lane_y(zu), &dpt, &deta, &dm);
  g[0] = ev_out(dpt, ev_off_pt());
  g[1] = ev_out(deta, ev_off_angle(ew));
  g[2] = ev_out(vp, ev_off_angle(ew));
  g[3] = ev_out(dm, ev_off_pt());
}

// g dm/dp of both legs of every pair: ga, gb (n, 4).
extern "C" void egh_pairs(const double *a, const double *b, const double *g, int64_t n, double *ga,
                          double *gb, uint8_t *ok) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i++) {
    const double *x = a + 4 * i, *y = b + 4 * i;
    const uint32_t wmax = umax32(word(x), word(y)), ew = wmax & 0x7ff00000u;
    EvPart p, q;
    EvGrad o;
    ff mp, mq;
    ok[i] = stage(x, wmax, T, &p, &mp) && stage(y, wmax, T, &q, &mq) && ev_pair_grad(p, q, g[i], T, &o);
    for (int k = 0; k < 4; k++) ga[4 * i + k] = gb[4 * i + k] = NAN;
    if (!ok[i]) continue;
    leg_out(p, mp, ew, T, o.we, o.zu, o.vp, ga + 4 * i);
    leg_out(q, mq, ew, T, neg(o.we), o.zu, neg(o.vp), gb + 4 * i);
  }
}

// J^T gs of every particle: out (n, 4).  Two particles at a time, as the kernel takes them (n even).
extern "C" void egh_sums(const double *v, const double *gs, int64_t n, double *out, uint8_t *ok) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i += 2) {
    EvPart p[2];
    EvOwn<ff> o[2];
    ff g[2][4], mm;
    uint32_t ew[2], eg[2];
    for (int l = 0; l < 2; l++) {
      const double *x = v + 4 * (i + l), *s = gs + 4 * (i + l);
      ew[l] = word(x) & 0x7ff00000u;
      ok[i + l] = stage(x, word(x), T, &p[l], &mm);
      o[l] = ev_own(p[l], mm);
      eg[l] = ev_gs(s[0], s[1], s[2], s[3], g[l]);
      ok[i + l] = ok[i + l] && eg[l] != 1u;
    }
    const EvOwn<ff2> O = pack(o[0], o[1]);
    ff2 G[4], t[4];
    for (int k = 0; k < 4; k++) G[k] = pack(g[0][k], g[1][k]);
    ev_sum_terms(O, ev_leg(O, T), G, T, t);
    for (int l = 0; l < 2; l++)
      for (int k = 0; k < 4; k++)
        out[4 * (i + l) + k] = ev_out(l ? lane_y(t[k]) : lane_x(t[k]),
                                      k == 0 || k == 3 ? ev_off_gs_pt(eg[l]) : ev_off_gs_angle(eg[l], ew[l]));
  }
}
