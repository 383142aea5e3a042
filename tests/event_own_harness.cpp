// Host build of a staged particle's own terms (paper_2312_02756_gb300/csrc/event_lc.cuh,
// event_lc_grad.cuh) as the jagged kernels form them: Cartesian components, and J^T gs one particle at
// a time.
#include <math.h>
#include <stdint.h>

#include "../paper_2312_02756_gb300/csrc/event_lc_grad.cuh"

using namespace gvx::ffm;

static uint32_t word(const double *v) { return umax32(dhi(v[0]), dhi(v[3]) & 0x7fffffffu); }

static bool in_domain(const double *v) {
  return lc_in_domain(dhi(v[0]), dhi(v[3]) & 0x7fffffffu, dhi(v[1]) & 0x7fffffffu, dhi(v[2]) & 0x7fffffffu, word(v));
}

// (px, py, pz, E) of every particle: out (n, 4).
extern "C" void eoh_cart(const double *v, int64_t n, double *out, uint8_t *ok) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i++) {
    const double *x = v + 4 * i;
    if (!(ok[i] = in_domain(x))) continue;
    const uint32_t rb = (word(x) & 0x7ff00000u) - (127u << 20);
    const ff pt = cvt1(cvt_parts(dhi(x[0]), dlo(x[0]), rb));
    const ff m = cvt1(cvt_parts(dhi(x[3]) & 0x7fffffffu, dlo(x[3]), rb));
    uint32_t ne, np;
    const ff re = own_reduce(x[1], angle_fx(x[1]), &ne), rp = own_reduce(x[2], angle_fx(x[2]), &np);
    ff sh, sn, cs;
    const LcLeg<ff> L = lc_leg_at(pt, m, re, &ne, T.hyp, &sh);
    sincos_lc_at(rp, np, T.sin, &sn, &cs);
    out[4 * i] = lc_to_double(lc_mul(pt, cs), rb);
    out[4 * i + 1] = copysign(1.0, x[2]) * lc_to_double(lc_mul(pt, sn), rb);
    out[4 * i + 2] = copysign(1.0, x[1]) * lc_to_double(lc_mul(pt, sh), rb);
    out[4 * i + 3] = lc_to_double(L.E, rb);
  }
}

// J^T gs of every particle: out (n, 4).
extern "C" void eoh_sums(const double *v, const double *gs, int64_t n, double *out, uint8_t *ok) {
  const LcTab T{kHypTab, kSinTab};
  for (int64_t i = 0; i < n; i++) {
    const double *x = v + 4 * i, *s = gs + 4 * i;
    ff g[4], t[4];
    const uint32_t ew = word(x) & 0x7ff00000u, rb = ew - (127u << 20), eg = ev_gs(s[0], s[1], s[2], s[3], g);
    if (!(ok[i] = in_domain(x) && eg > 1u)) continue;
    EvPart p;
    const ff pt = cvt1(cvt_parts(dhi(x[0]), dlo(x[0]), rb));
    const ff m = cvt1(cvt_parts(dhi(x[3]) & 0x7fffffffu, dlo(x[3]), rb));
    p.eta = angle_fx(x[1]);
    p.phi = angle_fx(x[2]);
    uint32_t ne;
    const ff re = fx_half_reduce(2 * p.eta, &ne);
    const LcLeg<ff> L = lc_leg_at(pt, m, re, &ne, T.hyp);
    p.dy = gvx_f4{L.D.hi, L.Y.hi, L.D.lo, L.Y.lo};
    p.pt_hi = pt.hi;
    p.pt_lo = pt.lo;
    EvOwn<ff> own = ev_own(p, with_sign(m, dhi(x[3])));
    own.re = own_reduce(x[1], p.eta, &own.n[0]);
    own.rp = own_reduce(x[2], p.phi, &own.j[0]);
    ev_sum_terms(own, ev_leg(own, T), g, T, t);
    for (int k = 0; k < 4; k++)
      out[4 * i + k] = ev_out(t[k], k == 0 || k == 3 ? ev_off_gs_pt(eg) : ev_off_gs_angle(eg, ew));
  }
}
