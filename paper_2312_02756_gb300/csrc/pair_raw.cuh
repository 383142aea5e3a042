// One FP64 pair mass from the raw values of its particles: the elementwise kernel, and the pairs
// that the event kernels leave to it.
#pragma once

#include "mass_lc.cuh"
#include "pair_math.cuh"

namespace gvx {

// The light-cone float-float fast path (mass_lc.cuh), the FP64 formulas outside its domain.
__device__ __forceinline__ double pair_mass_raw(const V4<double> &x, const V4<double> &y,
                                                const ffm::LcTab &T) {
  double m;
  if (!ffm::pair_mass_lc(x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w, T, &m))
    m = sqrt(pair_terms(make_leg(x), make_leg(y)).m2);
  return m;
}

// The same for two particles of an event, out of line: the event kernels' loops take it for the
// rare pairs outside the float-float domain, and inline it would cost them registers.
template <int LP>
__device__ __noinline__ double pair_mass_at(const void *c0, const void *c1, const void *c2,
                                            const void *c3, int64_t i, int64_t j) {
  const Lv p = {{c0, c1, c2, c3}, LP};
  return pair_mass_raw(ld4c<LP>(p, i), ld4c<LP>(p, j), ffm::LcTab{ffm::kHypTab, ffm::kSinTab});
}

}  // namespace gvx
