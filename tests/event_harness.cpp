// Host build of the event kernels' staged pair (paper_2312_02756_gb300/csrc/event_lc.cuh): the same
// source the kernels compile, called over arrays of pairs.
#include <math.h>
#include <stdint.h>

#include "../paper_2312_02756_gb300/csrc/event_lc.cuh"

using namespace gvx::ffm;

static bool stage(const double *v, uint32_t wmax, const LcTab &T, EvPart *p) {
  const uint32_t hp = dhi(v[0]), hm = dhi(v[3]) & 0x7fffffffu;
  if (!lc_in_domain(hp, hm, dhi(v[1]) & 0x7fffffffu, dhi(v[2]) & 0x7fffffffu, wmax)) return false;
  const uint32_t ew = wmax & 0x7ff00000u, rb = ew - (127u << 20);
  const ff pt = cvt1(cvt_parts(hp, dlo(v[0]), rb)), m = cvt1(cvt_parts(hm, dlo(v[3]), rb));
  p->eta = angle_fx(v[1]);
  p->phi = angle_fx(v[2]);
  uint32_t n;
  const ff r = fx_half_reduce(2 * p->eta, &n);
  const LcLeg<ff> L = lc_leg_at(pt, m, r, &n, T.hyp);
  p->dy = gvx_f4{L.D.hi, L.Y.hi, L.D.lo, L.Y.lo};
  p->pt_hi = pt.hi;
  p->pt_lo = pt.lo;
  p->scale = ew;
  return true;
}

extern "C" void evh_pairs(const double *a, const double *b, int64_t n, double *m, uint8_t *ok) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i++) {
    const double *x = a + 4 * i, *y = b + 4 * i;
    const uint32_t wmax = umax32(umax32(dhi(x[0]), dhi(x[3]) & 0x7fffffffu),
                                 umax32(dhi(y[0]), dhi(y[3]) & 0x7fffffffu));
    EvPart p, q;
    ff m2s;
    ok[i] = stage(x, wmax, T, &p) && stage(y, wmax, T, &q) && ev_pair_m2(p, q, T, &m2s);
    m[i] = ok[i] ? lc_mass_out(m2s, wmax & 0x7ff00000u) : NAN;
  }
}
