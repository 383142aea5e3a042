// The jagged adjoint's pair terms as the kernel forms them, with the angles' FP64 differences at hand for
// the pairs whose staged ones do not give a small difference.
#include "event_grad_harness.cpp"

// leg_out with the particle's own small angles from their doubles.
static void leg_near(const double *x, const EvPart &p, const ff &m, uint32_t ew, const LcTab &T, const ff2 &we,
                     const ff2 &zu, const ff &vp, double *g) {
  EvOwn<ff> o = ev_own(p, m);
  if (fx_small(p.eta, p.phi)) {
    o.re = own_reduce(x[1], p.eta, &o.n[0]);
    o.rp = own_reduce(x[2], p.phi, &o.j[0]);
  }
  ff dpt, deta, dm;
  ev_grad_terms(o, ev_leg(o, T), lane_x(we), lane_y(we), lane_x(zu), lane_y(zu), &dpt, &deta, &dm);
  g[0] = ev_out(dpt, ev_off_pt());
  g[1] = ev_out(deta, ev_off_angle(ew));
  g[2] = ev_out(vp, ev_off_angle(ew));
  g[3] = ev_out(dm, ev_off_pt());
}

extern "C" void enh_pairs(const double *a, const double *b, const double *g, int64_t n, double *ga,
                          double *gb, uint8_t *ok, uint8_t *asked) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i++) {
    const double *x = a + 4 * i, *y = b + 4 * i;
    const uint32_t wmax = umax32(word(x), word(y)), ew = wmax & 0x7ff00000u;
    EvPart p, q;
    EvGrad o;
    ff mp, mq;
    for (int k = 0; k < 4; k++) ga[4 * i + k] = gb[4 * i + k] = NAN;
    ok[i] = asked[i] = 0;
    if (!stage(x, wmax, T, &p, &mp) || !stage(y, wmax, T, &q, &mq)) continue;
    const auto exact_words = [](const double *v) { return ev_exact(dhi(v[1]) & 0x7fffffffu, dhi(v[2]) & 0x7fffffffu); };
    const bool exact = exact_words(x) && exact_words(y);
    ok[i] = ev_pair_grad(p, q, exact, [&](double *d) {
      d[0] = x[1] - y[1];
      d[1] = x[2] - y[2];
      asked[i] = 1;
      return true;
    }, g[i], T, &o);
    if (!ok[i]) continue;
    leg_near(x, p, mp, ew, T, o.we, o.zu, o.vp, ga + 4 * i);
    leg_near(y, q, mq, ew, T, neg(o.we), o.zu, neg(o.vp), gb + 4 * i);
  }
}
