// Adjoint of the jagged-event pair masses and event sums (the per-event combinatorics of the
// RDataFrame analyses that GenVectorX names as its next target, Sec. 6, differentiated; the pair
// mass is that of Sec. 4.1, Fig. 1).
//
// For particle i of event e, with the upstream gradients gm of the packed pair masses and gs of
// the event sums (PxPyPzE):
//   grad_i = sum over j != i of gm[pair(i, j)] dm(p_i, p_j)/dp_i  +  J_i^T gs[e],
// J_i = d(px, py, pz, E)/d(pt, eta, phi, m) of the particle.
//
// CTAs take tiles of consecutive events (grid-stride over tiles) and deal a tile's events to their
// warps in batches of whole events of at most kCapW particles, as the forward kernel (jagged.cu)
// does; a warp that ends a batch draws the next one's number.  Per batch, one warp, with its own
// part of shared memory and no block barrier:
//   (a) per particle: its light-cone terms at its event's power of two and its angles in fixed point
//       (event_lc.cuh);
//   (b) in chunks of kPC pairs, one lane per pair: the five numbers of event_lc_grad.cuh, which
//       enter both legs' gradients with a sign only, into the pair's slot.  The pairs are taken by
//       their distance: row t of an event of n particles holds the pairs (i, i + t modulo n).  A
//       difference below 2^-12 between angles that are not exact in fixed point (one pair in 10^6) is
//       taken in FP64 from the particles at once: left to the second launch, such a pair costs that
//       launch 35 us of latency;
//   (c) after each chunk, one lane per particle: its signed sums over its pairs of the chunk, two per
//       row, in a fixed order, so that the result does not depend on scheduling and no atomic
//       operation touches it.  With the pairs in that order the lanes of an event read
//       neighbouring slots;
//   (d) per particle: its gradient from the sums, and J^T gs, both in float-float, converted by
//       integer operations and added in FP64; sinh(eta) and sin(phi) of an angle below 2^-12 from the
//       particle itself.
// What that leaves is noted in a word per tile in the workspace and done by a second launch: pairs
// outside the float-float domain (either particle outside the forward's domain at the event's scale
// or with pt = 0, directions near each other across phi = +-pi, a scaled m^2 below 2^-80, |gm|
// outside [2^-60, 2^20]) and event-sum parts with gs out of range, by walking the batches that met one
// once more and adding the FP64 formulas to the gradients written; and events with more than kCapW
// particles, by a CTA straight from global memory with the elementwise adjoint.  The pair offsets
// are those the forward call wrote; each tile checks them (and the offsets) against the event sizes
// and the pair count before it reads any pair gradient, and records GVX_ERR_OFFSETS where they do not
// match; of such a tile the second launch does the events whose own offsets are right, each by a CTA.
//
// Bound by issue (the first launch; 66% of the slots, held back by dependent chains at 20 warps per SM).
// 300,007 events, 9.6 M pairs: 395 us both launches (382 us before the small angles and differences of
// (b) and (d), which the figures below leave out), against 550 us for block-wide sub-batches whose
// particles walked their partners (seven sums of products per direction, 1,150 warp instructions per
// 32 pairs) and a second launch over every tile with a pair near 2 pi.  By step: pairs in packed
// order, whose lanes read slots far apart, 465 us; by distance 413; without a call in the first
// launch 392; chunks of 96 pairs and 5 CTAs per SM in place of 128 and 4 382 (64 pairs: 410).  Both
// particles of a lane on paired FP32 instructions in (d): 422 us (moves and spills).
#include <cuda_runtime.h>

#include "common.cuh"
#include "event_lc_grad.cuh"
#include "pair_math.cuh"

namespace gvx {
namespace {

constexpr int kNT = 128;    // threads per CTA
constexpr int kCtas = 5;    // CTAs per SM
constexpr int kTE = 128;    // events per tile at most
constexpr int kCapW = 64;   // particles per warp batch
constexpr int kPC = 96;     // pairs per chunk
constexpr int kRows = kCapW * (kCapW - 1) / 2 / 32 + 1;  // words of the row mask: a bit per pair
constexpr unsigned kAll = 0xffffffffu;
constexpr int kMinTE = 16;  // events per tile at least
constexpr int kWsEvents = 14;  // gvx_event_pair_masses_bwd_workspace: a word per kWsEvents events
static_assert(kMinTE >= kWsEvents, "the workspace holds a word per tile");

// One warp's part of shared memory.
struct __align__(16) WarpBuf {
  float4 dy[kCapW];       // (D.hi, Y.hi, D.lo, Y.lo)
  longlong2 ang[kCapW];   // (eta, phi), units of 2^-59
  float4 w0[kPC], w1[kPC];  // by pair of the chunk: lanes (W, Ve) and (Z, U); in a second walk the
  float2 w2[kPC];           // FP64 gradients by particle.  w2: Vp
  float2 pt[kCapW];       // pt; hi < 0: outside the float-float domain
  float2 mm[kCapW];       // m
  float2 sum[5][kCapW];   // W, Ve, Z, U, Vp summed over the chunks so far
  int4 info[32];          // by non-empty event: first particle, particles, first pair, event of the tile | first row << 8
  uint32_t scale[32];     // by non-empty event: the largest high word of pt and |m|
  int row[kCapW / 2];     // by row: its first pair, its event's first particle and size, the distance
  uint32_t rows[kRows];   // bit q: a row starts at pair q of the batch
};
static_assert(sizeof(float4) * 2 * kPC >= sizeof(V4<double>) * kCapW, "FP64 gradients in place of the slots");
constexpr size_t kDynSmem = (kNT / 32) * sizeof(WarpBuf);

struct BArgs {
  Lv p;
  const int64_t *off, *pair_off;
  int64_t n_events, n_particles, n_pairs;
  const double *gpm;
  Lv gsum;
  bool has_gsum;
  LvOut grad;
  int32_t *status;
  unsigned long long *left;  // workspace: a word per tile, what the first launch left of it
  int te;   // events per tile
  int cap;  // particles per batch (an event larger than it, up to kCapW, is a batch of its own)
};

// J^T gs in FP64 for one particle: gs = (gx, gy, gz, gE) against the rows
//   px: (cos phi, 0, -pt sin phi, 0)       py: (sin phi, 0, pt cos phi, 0)
//   pz: (sinh eta, pt cosh eta, 0, 0)      E:  (P cosh eta, P pt sinh eta, 0, m) / E,
// P = pt cosh eta; for a massless particle (E = P) the E row is (cosh eta, pt sinh eta, 0, 0).
__device__ __noinline__ V4<double> sum_part(V4<double> x, V4<double> gs) {
  const double pt = x.x, eta = x.y, phi = x.z, m = x.w;
  double s, c;
  sincos(phi, &s, &c);
  const double sh = sinh(eta), ch = cosh(eta);
  double eE0, eE1, eE3;  // E row: d/dpt, d/deta, d/dm
  if (m == 0.0) {
    eE0 = ch;
    eE1 = pt * sh;
    eE3 = 0.0;
  } else {
    const double P = pt * ch;
    const double E = sqrt(fma(P, P, m * m));
    eE0 = P * ch / E;
    eE1 = P * pt * sh / E;
    eE3 = m / E;
  }
  V4<double> g;
  g.x = fma(gs.x, c, fma(gs.y, s, fma(gs.z, sh, gs.w * eE0)));
  g.y = fma(gs.z, pt * ch, gs.w * eE1);
  g.z = pt * fma(gs.y, c, -gs.x * s);
  g.w = gs.w * eE3;
  return g;
}

// gm-weighted gradient of particle i's leg over its partners in one event, everything read from
// global memory (the path of events too large to stage).
template <int LP>
__device__ __forceinline__ void partners_from_global(const BArgs &A, const ffm::LcTab &T,
                                                     int64_t i, int64_t base, int64_t n,
                                                     int64_t pair0, double *acc) {
  const V4<double> x = ld4c<LP>(A.p, i);
  const int64_t li = i - base;
  for (int64_t lj = 0; lj < n; lj++) {
    if (lj == li) continue;
    const int64_t r = li < lj ? li : lj, q = li < lj ? lj : li;
    const double g = __ldg(A.gpm + pair0 + r * n - r * (r + 1) / 2 + (q - r - 1));
    const V4<double> y = ld4c<LP>(A.p, base + lj);
    double o[8];
    if (!ffm::pair_mass_grad_lc(x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w, g, false, 0.0, T, o)) {
      V4<double> g1, g2;
      pair_mass_grad(x, y, g, g1, g2);
      o[0] = g1.x;
      o[1] = g1.y;
      o[2] = g1.z;
      o[3] = g1.w;
    }
    for (int c = 0; c < 4; c++) acc[c] += o[c];
  }
}

// An event with more than kCapW particles: its particles in strides of the CTA, each against all its
// partners from global memory.
template <int LP, int LS, int LG>
__device__ __forceinline__ void big_event(const BArgs &A, const ffm::LcTab &T, int64_t e, int64_t pbeg,
                                       int64_t n, int64_t pair0) {
  for (int64_t t = threadIdx.x; t < n; t += kNT) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const V4<double> x = ld4c<LP>(A.p, pbeg + t);
    if (A.has_gsum) {
      const V4<double> sp = sum_part(x, ld4c<LS>(A.gsum, e));
      acc[0] = sp.x;
      acc[1] = sp.y;
      acc[2] = sp.z;
      acc[3] = sp.w;
    }
    partners_from_global<LP>(A, T, pbeg + t, pbeg, n, pair0, acc);
    st4<double, LG>(A.grad, pbeg + t, V4<double>{acc[0], acc[1], acc[2], acc[3]});
  }
}

// Whether a particle's angles are exact travels to the pairs as the last bit of D.lo, 2^-47 of a D that
// is good to 2^-45.
__device__ __forceinline__ float mark_inexact(float lo, bool inexact) {
  return __uint_as_float((__float_as_uint(lo) & ~1u) | (uint32_t)inexact);
}
__device__ __forceinline__ bool both_exact(const ffm::EvPart &a, const ffm::EvPart &b) {
  return ((__float_as_uint(a.dy.z) | __float_as_uint(b.dy.z)) & 1u) == 0u;
}

// (a) The particles of places c and c + 32 (the second only with `two`) at their events' scale words,
// as the lanes of paired FP32 instructions.  False where one lies outside the float-float domain.
__device__ __forceinline__ bool stage_particles(WarpBuf &W, int c, bool two, const V4<double> *x,
                                                const uint32_t *wmax, const ffm::LcTab &T) {
  bool ok[2], exact[2];
  ffm::ff pt[2], mm[2], re[2];
  int64_t ae[2], ap[2];
  uint32_t n[2];
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const uint32_t hp = ffm::dhi(x[r].x), hm = ffm::dhi(x[r].w) & 0x7fffffffu;
    const uint32_t he = ffm::dhi(x[r].y) & 0x7fffffffu, hf = ffm::dhi(x[r].z) & 0x7fffffffu;
    ok[r] = hp >= 0x100000u && ffm::lc_in_domain(hp, hm, he, hf, wmax[r]);
    exact[r] = ffm::ev_exact(he, hf);
    const uint32_t rb = (wmax[r] & 0x7ff00000u) - (127u << 20);
    pt[r] = ffm::cvt1(ffm::cvt_parts(hp, ffm::dlo(x[r].x), rb));
    mm[r] = ffm::cvt1(ffm::cvt_parts(hm, ffm::dlo(x[r].w), rb));
    ae[r] = ffm::angle_fx(x[r].y);
    ap[r] = ffm::angle_fx(x[r].z);
    re[r] = ffm::fx_half_reduce(2 * ae[r], &n[r]);
  }
  const ffm::LcLeg<ffm::ff2> L =
      ffm::lc_leg_at(ffm::pack(pt[0], pt[1]), ffm::pack(mm[0], mm[1]), ffm::pack(re[0], re[1]), n, T.hyp);
#pragma unroll
  for (int r = 0; r < 2; r++) {
    if (r == 1 && !two) break;
    const int k = c + 32 * r;
    const ffm::ff D = r ? ffm::lane_y(L.D) : ffm::lane_x(L.D), Y = r ? ffm::lane_y(L.Y) : ffm::lane_x(L.Y);
    const ffm::ff ms = ffm::with_sign(mm[r], ffm::dhi(x[r].w));
    W.dy[k] = make_float4(D.hi, Y.hi, mark_inexact(D.lo, !exact[r]), Y.lo);
    W.ang[k] = make_longlong2(ae[r], ap[r]);
    W.pt[k] = make_float2(ok[r] ? pt[r].hi : -1.0f, pt[r].lo);
    W.mm[k] = make_float2(ms.hi, ms.lo);
  }
  return ok[0] && (ok[1] || !two);
}

__device__ __forceinline__ ffm::EvPart staged(const WarpBuf &W, int c) {
  const longlong2 a = W.ang[c];
  const float2 t = W.pt[c];
  return ffm::EvPart{W.dy[c], a.x, a.y, t.x, t.y, 0u, 0u};
}

// a += x, the leading parts without error.
__device__ __forceinline__ void acc_add(ffm::ff2 &a, const ffm::ff2 &x) {
  const ffm::ff2 s = ffm::two_sum2(a.hi, x.hi);
  a = {s.hi, ffm::add2(a.lo, ffm::add2(s.lo, x.lo))};
}
__device__ __forceinline__ void acc_add(ffm::ff &a, const ffm::ff &x) {
  const ffm::ff s = ffm::two_sum(a.hi, x.hi);
  a = {s.hi, ffm::fadd(a.lo, ffm::fadd(s.lo, x.lo))};
}
struct Sums {
  ffm::ff2 we, zu;
  ffm::ff vp;
};
__device__ __forceinline__ void add_slot(Sums &s, const WarpBuf &W, int k) {
  const float4 a = W.w0[k], b = W.w1[k];
  const float2 v = W.w2[k];
  acc_add(s.we, ffm::ff2{ffm::mk2(a.x, a.y), ffm::mk2(a.z, a.w)});
  acc_add(s.zu, ffm::ff2{ffm::mk2(b.x, b.y), ffm::mk2(b.z, b.w)});
  acc_add(s.vp, ffm::ff{v.x, v.y});
}

// One batch by one warp: `take` events of the tile from event sb on (lane l < take having event
// sb + l with particles lo .. hi - 1), together at most kCapW particles.  RARE: a second walk, which
// adds what the first one left to the gradients written and nothing else.  Returns whether
// something was left.
template <int LP, int LS, int LG, bool RARE>
__device__ __forceinline__ bool warp_batch(const BArgs &A, const ffm::LcTab &T, WarpBuf &W, int64_t e0,
                                           int sb, int take, int64_t lo, int64_t hi, const int64_t *s_po) {
  const int lane = threadIdx.x & 31;
  const unsigned upto = 0xffffffffu >> (31 - lane), below = upto >> 1;
  const int64_t pb = __shfl_sync(kAll, lo, 0);
  const int np = (int)(__shfl_sync(kAll, hi, take - 1) - pb);
  const int64_t q0 = s_po[sb];
  const int total = (int)(s_po[sb + take] - q0);
  const double *const gpm = A.gpm + q0;
  V4<double> x[2] = {{0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0}};
#pragma unroll
  for (int r = 0; r < 2; r++)
    if (lane + 32 * r < np && GVX_IN_BOUNDS(pb + lane + 32 * r, A.n_particles, A.status))
      x[r] = ld4c<LP>(A.p, pb + lane + 32 * r);
  // non-empty events in order; the particles they start at as bits
  const int n_l = lane < take ? (int)(hi - lo) : 0, st_l = (int)(lo - pb);
  const unsigned nz = __ballot_sync(kAll, n_l > 0);
  const unsigned m0 = __reduce_or_sync(kAll, n_l > 0 && st_l < 32 ? 1u << st_l : 0u);
  const unsigned m1 = __reduce_or_sync(kAll, n_l > 0 && st_l >= 32 ? 1u << (st_l - 32) : 0u);
  int nrow = n_l >> 1;  // rows up to and with the lane's event
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kAll, nrow, o);
    if (lane >= o) nrow += t;
  }
  if (n_l > 0) {
    const int k = __popc(nz & below);
    W.info[k] = make_int4(st_l, n_l, (int)(s_po[sb + lane] - q0), (sb + lane) | (nrow - (n_l >> 1)) << 8);
    W.scale[k] = 0u;
  }
  for (int w = lane; w < kRows; w += 32) W.rows[w] = 0u;
  __syncwarp();
  int rank[2];
#pragma unroll
  for (int r = 0; r < 2; r++) {
    rank[r] = r ? __popc(m0) + __popc(m1 & upto) - 1 : __popc(m0 & upto) - 1;
    if (lane + 32 * r < np)
      atomicMax(&W.scale[rank[r]], ffm::umax32(ffm::dhi(x[r].x), ffm::dhi(x[r].w) & 0x7fffffffu));
  }
  __syncwarp();
  bool rare = false;
  uint32_t wmax[2] = {0u, 0u};
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const int c = lane + 32 * r;
    if (c < np) {
      const int4 v = W.info[rank[r]];
      const int li = c - v.x;
      if (li > 0 && 2 * li <= v.y) {  // row li: pairs (i, i + li), i from 0, at slots first + i
        const int first = v.z + (li - 1) * v.y;
        W.row[(v.w >> 8) + li - 1] = first | v.x << 11 | v.y << 17 | li << 24;
        atomicOr(&W.rows[first >> 5], 1u << (first & 31));
      }
      wmax[r] = W.scale[rank[r]];
    }
  }
  if (lane < np) rare = !stage_particles(W, lane, lane + 32 < np, x, wmax, T);
  V4<double> *const dg = reinterpret_cast<V4<double> *>(W.w0);  // RARE: FP64 gradients by particle
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const int c = lane + 32 * r;
    if constexpr (RARE) {
      dg[c] = {0.0, 0.0, 0.0, 0.0};
    } else {
#pragma unroll
      for (int k = 0; k < 5; k++) W.sum[k][c] = make_float2(0.0f, 0.0f);
    }
  }
  const bool extreme = __any_sync(kAll, rare);
  __syncwarp();  // the staged places and rows are visible to the warp (a vote orders no memory)
  int rows = -1;  // rows that start before the current word, less one
  for (int c0 = 0; c0 < total; c0 += kPC) {
    const int c1 = c0 + kPC < total ? c0 + kPC : total;
    // (b)
    for (int r0 = c0; r0 < c1; r0 += 32) {
      const unsigned w = W.rows[r0 >> 5];
      const int q = r0 + lane;
      int i = 0, j = 0;
      bool slow = false;
      double g = 0.0;
      if (q < c1) {
        const int rec = W.row[rows + __popc(w & upto)];
        const int first = rec & 0x7ff, base = (rec >> 11) & 0x3f, n = (rec >> 17) & 0x7f, t = rec >> 24;
        i = q - first;
        j = i + t < n ? i + t : i + t - n;
        const int a = min(i, j);  // its number in the packed order
        const int k = first - (t - 1) * n + a * n - (a * (a + 1) >> 1) + (max(i, j) - a - 1);
        if (GVX_IN_BOUNDS(q0 + k, A.n_pairs, A.status)) g = __ldg(gpm + k);
        i += base;
        j += base;
        if (GVX_IN_BOUNDS(i, np, A.status) && GVX_IN_BOUNDS(j, np, A.status)) {
          const ffm::EvPart a = staged(W, i), b = staged(W, j);
          ffm::EvGrad o;
          const auto near = [&](double *d) {
            const V4<double> u = ld4c<LP>(A.p, pb + i), v = ld4c<LP>(A.p, pb + j);
            d[0] = u.y - v.y;
            d[1] = u.z - v.z;
            return true;
          };
          slow = !ffm::ev_pair_grad(a, b, both_exact(a, b), near, g, T, &o) ||
                 (extreme && (a.pt_hi < 0.0f || b.pt_hi < 0.0f));
          if constexpr (!RARE) {
            if (slow) {
              o = ffm::EvGrad{{ffm::bc2(0.0f), ffm::bc2(0.0f)}, {ffm::bc2(0.0f), ffm::bc2(0.0f)}, {0.0f, 0.0f}};
              rare = true;
            }
            W.w0[q - c0] = make_float4(o.we.hi.x, o.we.hi.y, o.we.lo.x, o.we.lo.y);
            W.w1[q - c0] = make_float4(o.zu.hi.x, o.zu.hi.y, o.zu.lo.x, o.zu.lo.y);
            W.w2[q - c0] = make_float2(o.vp.hi, o.vp.lo);
          }
        }
      }
      rows += __popc(w);
      if constexpr (RARE) {  // the pairs left, their gradients added in the pairs' order
        V4<double> g1 = {0, 0, 0, 0}, g2 = {0, 0, 0, 0};
        if (slow) pair_mass_grad(ld4c<LP>(A.p, pb + i), ld4c<LP>(A.p, pb + j), g, g1, g2);
        for (unsigned left = __ballot_sync(kAll, slow); left; left &= left - 1) {
          if (lane == __ffs((int)left) - 1) {
            V4<double> t = dg[i];
            dg[i] = {t.x + g1.x, t.y + g1.y, t.z + g1.z, t.w + g1.w};
            t = dg[j];
            dg[j] = {t.x + g2.x, t.y + g2.y, t.z + g2.z, t.w + g2.w};
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    // (c)
    if constexpr (!RARE) {
#pragma unroll 1
      for (int r = 0; r < 2; r++) {
        const int c = lane + 32 * r;
        if (c >= np) break;
        const int4 v = W.info[r ? rank[1] : rank[0]];
        const int n = v.y, li = c - v.x;
        if (v.z >= c1 || v.z + (n * (n - 1) >> 1) <= c0) continue;
        Sums s;
        {
          const float2 a = W.sum[0][c], b = W.sum[1][c], d = W.sum[2][c], e = W.sum[3][c], f = W.sum[4][c];
          s.we = {ffm::mk2(a.x, b.x), ffm::mk2(a.y, b.y)};
          s.zu = {ffm::mk2(d.x, e.x), ffm::mk2(d.y, e.y)};
          s.vp = {f.x, f.y};
        }
        // row t: pair (li, li + t) at the row's place li, and (li - t, li) at place li - t, modulo n;
        // the last row of an even n holds each of its n / 2 pairs once
        Sums o = {{ffm::bc2(0.0f), ffm::bc2(0.0f)}, {ffm::bc2(0.0f), ffm::bc2(0.0f)}, {0.0f, 0.0f}};
        const int len = c1 - c0;
        int t = c0 > v.z ? (c0 - v.z) / n + 1 : 1;
        for (int f = v.z + (t - 1) * n - c0; 2 * t <= n && f < len; t++, f += n) {
          const int in = li >= t ? li - t : li - t + n, last = 2 * t == n ? t : n;
          if (li < last && (unsigned)(f + li) < (unsigned)len) add_slot(s, W, f + li);
          if (in < last && (unsigned)(f + in) < (unsigned)len) add_slot(o, W, f + in);
        }
        acc_add(s.we, ffm::neg(o.we));
        acc_add(s.zu, o.zu);
        acc_add(s.vp, ffm::neg(o.vp));
        W.sum[0][c] = make_float2(s.we.hi.x, s.we.lo.x);
        W.sum[1][c] = make_float2(s.we.hi.y, s.we.lo.y);
        W.sum[2][c] = make_float2(s.zu.hi.x, s.zu.lo.x);
        W.sum[3][c] = make_float2(s.zu.hi.y, s.zu.lo.y);
        W.sum[4][c] = make_float2(s.vp.hi, s.vp.lo);
      }
      __syncwarp();  // before the next chunk overwrites the slots
    }
  }
  // (d)
#pragma unroll 1
  for (int r = 0; r < 2; r++) {
    const int c = lane + 32 * r;
    if (!(c < np && GVX_IN_BOUNDS(pb + c, A.n_particles, A.status))) break;
    const int k = r ? rank[1] : rank[0];
    const ffm::EvPart p = staged(W, c);
    const float2 m = W.mm[c];
    const uint32_t ew = W.scale[k] & 0x7ff00000u;
    const V4<double> g64 = A.has_gsum ? ld4c<LS>(A.gsum, e0 + (W.info[k].w & 0xff)) : V4<double>{0.0, 0.0, 0.0, 0.0};
    ffm::ff gs[4];
    const uint32_t ewg = ffm::ev_gs(g64.x, g64.y, g64.z, g64.w, gs);
    const bool fast = p.pt_hi >= 0.0f, done = !A.has_gsum || (fast && ewg != 1u);
    if constexpr (!RARE) {
      ffm::EvOwn<ffm::ff> own = ffm::ev_own(p, ffm::ff{m.x, m.y});
      if (__builtin_expect(ffm::fx_small(p.eta, p.phi), 0)) {  // the angles themselves, seldom
        const V4<double> v = ld4c<LP>(A.p, pb + c);
        own.re = ffm::own_reduce(v.y, p.eta, &own.n[0]);
        own.rp = ffm::own_reduce(v.z, p.phi, &own.j[0]);
      }
      const ffm::EvLeg<ffm::ff> l = ffm::ev_leg(own, T);
      const float2 s0 = W.sum[0][c], s1 = W.sum[1][c], s2 = W.sum[2][c], s3 = W.sum[3][c], s4 = W.sum[4][c];
      ffm::ff dpt, deta, dm;
      ffm::ev_grad_terms(own, l, ffm::ff{s0.x, s0.y}, ffm::ff{s1.x, s1.y}, ffm::ff{s2.x, s2.y},
                         ffm::ff{s3.x, s3.y}, &dpt, &deta, &dm);
      V4<double> o = {ffm::ev_out(dpt, ffm::ev_off_pt()), ffm::ev_out(deta, ffm::ev_off_angle(ew)),
                      ffm::ev_out(ffm::ff{s4.x, s4.y}, ffm::ev_off_angle(ew)), ffm::ev_out(dm, ffm::ev_off_pt())};
      if (ewg > 1u) {
        ffm::ff t[4];
        ffm::ev_sum_terms(own, l, gs, T, t);
        const uint32_t ep = ffm::ev_off_gs_pt(ewg), ea = ffm::ev_off_gs_angle(ewg, ew);
        o = {o.x + ffm::ev_out(t[0], ep), o.y + ffm::ev_out(t[1], ea), o.z + ffm::ev_out(t[2], ea),
             o.w + ffm::ev_out(t[3], ep)};
      }
      if (!fast) o = {0.0, 0.0, 0.0, 0.0};
      rare |= !done;
      st4<double, LG>(A.grad, pb + c, o);
    } else {
      V4<double> add = dg[c];
      if (!done) {
        const V4<double> sp = sum_part(ld4c<LP>(A.p, pb + c), g64);
        add = {add.x + sp.x, add.y + sp.y, add.z + sp.z, add.w + sp.w};
      }
      if (add.x != 0.0 || add.y != 0.0 || add.z != 0.0 || add.w != 0.0) {
        // plain coherent loads: the first launch wrote the array
        const V4<double> was = ld4<double, LG>(
            Lv{{A.grad.c[0], A.grad.c[1], A.grad.c[2], A.grad.c[3]}, A.grad.layout}, pb + c);
        st4<double, LG>(A.grad, pb + c, V4<double>{was.x + add.x, was.y + add.y, was.z + add.z, was.w + add.w});
      }
    }
  }
  rare = __any_sync(kAll, rare);
  __syncwarp();  // the buffer may be overwritten
  return rare;
}

// What one walk over a tile's batches shares among the warps.
struct TileState {
  int next;       // the next batch to take
  unsigned rare;  // bit b: a batch of number b modulo 32 left something
};

// The tile's batches: in the first walk every warp takes one after another by number, in the second
// the flagged ones are dealt out in turn.  *large: an event was left to the CTA.
template <int LP, int LS, int LG, bool RARE>
__device__ __forceinline__ void walk_tile(const BArgs &A, const ffm::LcTab &T, WarpBuf &W, TileState &S,
                                          int64_t e0, int ne, const int64_t *s_off, const int64_t *s_po,
                                          bool *large) {
  const int lane = threadIdx.x & 31;
  int mine = threadIdx.x >> 5, flagged = 0;
  for (int sb = 0, number = 0; sb < ne;) {
    const int64_t lo = s_off[min(sb + lane, ne)], hi = s_off[min(sb + lane + 1, ne)];
    const int64_t pb = __shfl_sync(kAll, lo, 0);
    int take = __popc(__ballot_sync(kAll, sb + lane < ne && hi - pb <= A.cap));
    if (take == 0) {
      if (__shfl_sync(kAll, hi, 0) - pb > kCapW) {
        *large = true;
        sb++;
        continue;
      }
      take = 1;
    }
    bool here;
    if constexpr (RARE) {
      const bool f = (S.rare >> (number & 31)) & 1u;
      here = f && (flagged & (kNT / 32 - 1)) == mine;
      flagged += f;
    } else {
      here = number == mine;
    }
    if (here) {
      const bool rare = warp_batch<LP, LS, LG, RARE>(A, T, W, e0, sb, take, lo, hi, s_po);
      if constexpr (!RARE) {
        int t = 0;
        if (lane == 0) {
          if (rare) atomicOr(&S.rare, 1u << (number & 31));
          t = atomicAdd(&S.next, 1);
        }
        mine = __shfl_sync(kAll, t, 0);
      }
    }
    number++;
    sb += take;
  }
}

constexpr unsigned long long kLarge = 1ull << 32, kBad = 2ull << 32;

// Whether the offsets of event e (particles a .. b - 1, pairs pa .. pb - 1) cannot be right.
__device__ __forceinline__ bool bad_event(const BArgs &A, int64_t e, int64_t a, int64_t b, int64_t pa, int64_t pb) {
  const int64_t n = b - a;
  return a < 0 || n < 0 || b > A.n_particles || n > (1ll << 31) || pa < 0 || pb > A.n_pairs ||
         pb - pa != n * (n - 1) / 2 || (e == 0 && (a != 0 || pa != 0));
}

// A tile's offsets into shared memory; false for a tile with an event whose offsets cannot be right.
__device__ __forceinline__ bool load_tile(const BArgs &A, int64_t e0, int ne, int64_t *s_off, int64_t *s_po) {
  for (int k = threadIdx.x; k <= ne; k += kNT) {
    s_off[k] = A.off[e0 + k];
    s_po[k] = A.pair_off[e0 + k];
  }
  __syncthreads();
  const int t = threadIdx.x;
  return !__syncthreads_or(t < ne && bad_event(A, e0 + t, s_off[t], s_off[t + 1], s_po[t], s_po[t + 1]));
}

template <int LP, int LS, int LG>
__global__ void __launch_bounds__(kNT, kCtas) event_pairs_bwd_kernel(const __grid_constant__ BArgs A) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  WarpBuf *bufs = reinterpret_cast<WarpBuf *>(s_dyn);
  __shared__ int64_t s_off[kTE + 1], s_po[kTE + 1];
  __shared__ TileState s_tile;
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};
  const int64_t n_tiles = (A.n_events + A.te - 1) / A.te;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t e0 = tile * A.te;
    const int ne = (int)(A.n_events - e0 < A.te ? A.n_events - e0 : A.te);
    __syncthreads();  // the previous tile is done with the shared arrays
    if (threadIdx.x == 0) s_tile = {kNT / 32, 0u};
    unsigned long long left = 0;
    if (load_tile(A, e0, ne, s_off, s_po)) {
      bool large = false;
      walk_tile<LP, LS, LG, false>(A, T, bufs[threadIdx.x >> 5], s_tile, e0, ne, s_off, s_po, &large);
      __syncthreads();
      left = s_tile.rare | (large ? kLarge : 0ull);
    } else {
      left = kBad;
      if (threadIdx.x == 0) raise_status(A.status, GVX_ERR_OFFSETS);
    }
    if (threadIdx.x == 0) A.left[tile] = left;
  }
}

// What the first launch left (nothing, most of the time): every block scans its share of the tiles'
// words and takes what they note.  A launch of its own, because a call anywhere in the first kernel
// costs its batches spills (413 us against 392 us at 300,007 events).  A tile counts kParts times, for
// its flagged batches and for every kParts-th of its large events, so that a few tiles of large events
// still reach all SMs (2,000 events of 150 particles: 2,284 us, by whole tiles 6,809 us).
constexpr int kParts = 8;

template <int LP, int LS, int LG>
__global__ void __launch_bounds__(kNT, 4) event_pairs_bwd_left_kernel(const __grid_constant__ BArgs A) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  WarpBuf *bufs = reinterpret_cast<WarpBuf *>(s_dyn);
  __shared__ int64_t s_off[kTE + 1], s_po[kTE + 1];
  __shared__ TileState s_tile;
  __shared__ unsigned long long s_left[kNT];
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};
  const int64_t n_tiles = (A.n_events + A.te - 1) / A.te;
  // the block's share: every gridDim.x-th, a thread looking at one (so that neighbouring tiles, often
  // alike, go to different blocks)
  for (int64_t t0 = blockIdx.x; t0 < kParts * n_tiles; t0 += (int64_t)gridDim.x * kNT) {
    const int64_t t = t0 + (int64_t)gridDim.x * threadIdx.x;
    unsigned long long mine = t < kParts * n_tiles ? A.left[t % n_tiles] : 0ull;
    if (t >= n_tiles) mine &= kLarge | kBad;  // the batches are part 0's
    if (!__syncthreads_or(mine != 0ull)) continue;
    s_left[threadIdx.x] = mine;
    __syncthreads();
    for (int k = 0; k < kNT; k++) {
      const unsigned long long left = s_left[k];
      if (left == 0ull) continue;
      const int64_t item = t0 + (int64_t)gridDim.x * k, e0 = item % n_tiles * A.te;
      const int ne = (int)(A.n_events - e0 < A.te ? A.n_events - e0 : A.te);
      __syncthreads();  // the previous tile is done with the shared arrays
      if (threadIdx.x == 0) s_tile = {0, (unsigned)left};
      load_tile(A, e0, ne, s_off, s_po);
      bool large;
      if ((unsigned)left != 0u)
        walk_tile<LP, LS, LG, true>(A, T, bufs[threadIdx.x >> 5], s_tile, e0, ne, s_off, s_po, &large);
      if (left & (kLarge | kBad))
        for (int e = (int)(item / n_tiles); e < ne; e += kParts) {
          const int64_t pbeg = s_off[e], n = s_off[e + 1] - pbeg;
          // of a tile with malformed offsets, every event whose own are right
          if ((left & kBad) ? !bad_event(A, e0 + e, pbeg, pbeg + n, s_po[e], s_po[e + 1]) : n > kCapW)
            big_event<LP, LS, LG>(A, T, e0 + e, pbeg, n, s_po[e]);
        }
    }
    __syncthreads();
  }
}

// Events per tile and particles per batch: whole tiles of kTE where they make kTileWaves per CTA that
// fits at once, smaller ones below (100,000 events: 143 us at 4 waves, 147 at 2, 167 at 1), and at the
// last step smaller batches, so that more warps share them (20,000 events: 46 us, with whole batches 48).
constexpr int kTileWaves = 4;
void tile_shape(int64_t n_events, int *te, int *cap) {
  const int64_t ctas = (int64_t)num_sms() * kCtas * kTileWaves;
  *te = kTE;
  *cap = kCapW;
  while (*te > kMinTE && n_events < *te * ctas) *te /= 2;
  if (*te == kMinTE) *cap = 32;
}

template <int LP, int LS, int LG>
cudaError_t launch_l(BArgs A, cudaStream_t s) {
  constexpr auto k = event_pairs_bwd_kernel<LP, LS, LG>, left = event_pairs_bwd_left_kernel<LP, LS, LG>;
  cudaError_t err =
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynSmem);
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(left, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynSmem);
  if (err != cudaSuccess) return err;
  tile_shape(A.n_events, &A.te, &A.cap);
  const int64_t n_tiles = (A.n_events + A.te - 1) / A.te;
  k<<<balanced_grid_of<k>(kNT, kDynSmem, n_tiles, 1), kNT, kDynSmem, s>>>(A);  // one tile per CTA and pass
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  left<<<balanced_grid_of<left>(kNT, kDynSmem, kParts * n_tiles, 1, 1), kNT, kDynSmem, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

size_t event_pairs_bwd_workspace(int64_t n_events) {
  return 256 + (size_t)((n_events + kWsEvents - 1) / kWsEvents) * sizeof(unsigned long long);
}

cudaError_t launch_event_pairs_bwd(const Lv &p, const int64_t *off, const int64_t *pair_off,
                                   int64_t n_events, int64_t n_particles, const double *gpm,
                                   int64_t n_pairs, const Lv *gsum, const LvOut &grad, void *ws,
                                   cudaStream_t s) {
  BArgs A;
  A.p = p;
  A.off = off;
  A.pair_off = pair_off;
  A.n_events = n_events;
  A.n_particles = n_particles;
  A.n_pairs = n_pairs;
  A.gpm = gpm;
  A.has_gsum = gsum != nullptr;
  A.gsum = gsum ? *gsum : Lv{{nullptr, nullptr, nullptr, nullptr}, GVX_SOA};
  A.grad = grad;
  A.status = device_status_word();
  A.left = (unsigned long long *)ws;
  const int lp = p.layout, ls = A.gsum.layout, lg = grad.layout;
  if (lp == GVX_SOA) {
    if (ls == GVX_SOA) return lg == GVX_SOA ? launch_l<GVX_SOA, GVX_SOA, GVX_SOA>(A, s)
                                            : launch_l<GVX_SOA, GVX_SOA, GVX_AOS>(A, s);
    return lg == GVX_SOA ? launch_l<GVX_SOA, GVX_AOS, GVX_SOA>(A, s)
                         : launch_l<GVX_SOA, GVX_AOS, GVX_AOS>(A, s);
  }
  if (ls == GVX_SOA) return lg == GVX_SOA ? launch_l<GVX_AOS, GVX_SOA, GVX_SOA>(A, s)
                                          : launch_l<GVX_AOS, GVX_SOA, GVX_AOS>(A, s);
  return lg == GVX_SOA ? launch_l<GVX_AOS, GVX_AOS, GVX_SOA>(A, s)
                       : launch_l<GVX_AOS, GVX_AOS, GVX_AOS>(A, s);
}

}  // namespace gvx
