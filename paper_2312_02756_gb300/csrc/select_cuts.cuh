// The selection's cuts pt >= pt_min and |eta| <= eta_max on the bits of the doubles (an FP64 comparison
// holds the FP64 pipe like an addition).
#pragma once

#include <math.h>

#include "ff.cuh"

namespace gvx {

// The doubles as integers of the same order: NaN beyond the infinity of its sign, -0 next below 0.
GVX_HD int64_t ordered_bits(double x) {
  const int64_t b = (int64_t)ffm::d2u(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

struct Cuts {
  int64_t pt_lo;     // pt's integer lies in [pt_lo, pt_lo + pt_span]: at least pt_min, at most infinity
  uint64_t pt_span;
  uint64_t eta_end;  // |eta|'s bits are below this
};

// -0 passes a threshold of 0, nothing passes a NaN.
inline Cuts make_cuts(double pt_min, double eta_max) {
  Cuts c;
  c.pt_lo = ordered_bits(pt_min == 0.0 ? -0.0 : pt_min);
  c.pt_span = (uint64_t)ordered_bits(INFINITY) - (uint64_t)c.pt_lo;
  c.eta_end = eta_max >= 0.0 ? (uint64_t)ordered_bits(fabs(eta_max)) + 1u : 0u;
  if (!(pt_min <= INFINITY)) c.eta_end = 0u;
  return c;
}

// The difference wraps around in unsigned arithmetic: two integers of opposite signs can lie more than
// 2^63 apart.
GVX_HD bool passes(double pt, double eta, const Cuts &c) {
  const uint64_t e = ffm::d2u(eta) & 0x7fffffffffffffffull;
  return (uint64_t)ordered_bits(pt) - (uint64_t)c.pt_lo <= c.pt_span && e < c.eta_end;
}

}  // namespace gvx
