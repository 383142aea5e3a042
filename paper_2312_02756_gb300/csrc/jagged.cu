// Jagged events: every in-event pair mass and every per-event summed 4-vector, in one
// persistent launch (the per-event combinatorics of the RDataFrame analyses that GenVectorX
// names as its next target, Sec. 6; the pair mass itself is that of Sec. 4.1, Fig. 1).
//
// Work unit: a tile of TE consecutive events.  CTAs take tiles in increasing order from an
// atomic counter and stay resident until the tiles run out.  Per tile:
//   1. load and validate offsets[e0 .. e0+TE];  n_e(n_e-1)/2 pairs per event, block scan;
//   2. decoupled look-back over the tile descriptors, 32 at a time, for the number of pairs before
//      the tile (bounded wait: a predecessor that never publishes makes the CTA record
//      GVX_ERR_TIMEOUT and go on);  write pair_offsets;
//   3. the tile's events in batches of whole events of at most kCapW particles, each batch by one
//      warp with its own part of shared memory and no block barrier: per particle once, the
//      float-float light-cone terms of its leg (pt, Y = E + P, D = m^2 / Y at its event's power of
//      two), its angles in fixed point (event_lc.cuh) and its Cartesian components in float-float;
//      then the event sums (two components per lane as the lanes of paired FP32 instructions, the
//      event's particles split over two lanes) and the pair masses, one lane per pair over the
//      batch's flattened pairs, coalesced stores.  A pair finds its particles from a bit mask of
//      the rows' first pairs (a row: one particle with its later partners): one popcount and one
//      row record instead of a search for the event and a decoding of the index.
//   4. What the batches leave is done after them, in a function of its own at the end of the tile (a
//      call inside the batches costs them spills): pairs outside the float-float domain (near-equal
//      directions, extreme particles), by walking the tile's batches once more and giving those
//      pairs the elementwise arithmetic; and events with more than kCapW particles, by the whole CTA,
//      staged the same way up to kCP particles, straight from global memory beyond.
// Tile descriptors are 64-bit words: 2 flag bits (aggregate / inclusive prefix) + 62-bit value.
//
// Bound by issue and the shared-memory/L1 data pipe together (445 warp instructions and 104 data
// wavefronts per 32 pairs, of which the two table gathers take about 40).  2^20 events, 33.5 M
// pairs: 0.56 ms a call, against 0.744 ms for block-wide sub-batches with FP64 angle differences
// and a search per pair (620 instructions per 32 pairs, FP64 pipe 35% busy).  Six CTAs of 128
// threads per SM (80 registers): eight (64 registers, 0.623 ms) leave the tables too little L1.
// Tiles of 64 events on 128 threads: 0.615 ms; 256 on 256: 0.587 ms.
#include <cuda_runtime.h>

#include <type_traits>

#include "common.cuh"
#include "event_lc.cuh"
#include "pair_index.cuh"
#include "pair_raw.cuh"

namespace gvx {
namespace {

constexpr int kCapW = 64;  // particles per warp batch
constexpr int kCP = 224;   // particles of an event that the CTA stages
constexpr int kRows = kCapW * (kCapW - 1) / 2 / 32 + 1;  // words of the row mask: a bit per pair
constexpr unsigned kAll = 0xffffffffu;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagInc = 2ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1;
constexpr unsigned long long kWaitLimitNs = 1000000000ull;  // 1 s bound on a look-back wait
constexpr unsigned long long kMaxPolls = 1ull << 26;        // backstop if the timer stalls
constexpr size_t kWsHeader = 256;                           // tile counter, padded
constexpr int kMinTE = 64;

// Staged particles: of one batch of a warp, or of one event by the CTA.  An array per member: the
// lanes of a pair loop read neighbouring partners, and whole records 64 bytes apart put four of them on
// the same banks (0.583 ms; 0.564 ms so).
struct Staged {
  float4 *dy;       // (D.hi, Y.hi, D.lo, Y.lo)
  longlong2 *ang;   // (eta, phi), units of 2^-59
  float4 *c0, *c1;  // (px, py) and (pz, E): float-float as (hi, hi, lo, lo), or two doubles
  float2 *pt;
  uint32_t *scale;  // the event's scale field, or 0: outside the float-float domain
  __device__ __forceinline__ ffm::EvPart part(int c) const {
    const longlong2 a = ang[c];
    const float2 t = pt[c];
    return ffm::EvPart{dy[c], a.x, a.y, t.x, t.y, scale[c], 0u};
  }
};
constexpr size_t kStagedBytes = 3 * sizeof(float4) + sizeof(longlong2) + sizeof(float2) + sizeof(uint32_t);

// One warp's part of shared memory.
struct __align__(16) WarpBuf {
  float4 dy[kCapW];
  longlong2 ang[kCapW];
  float4 c0[kCapW], c1[kCapW];
  float2 pt[kCapW];
  uint32_t sc[kCapW];
  int4 info[32];  // by non-empty event: first particle, particles, first pair, event of the tile
  uint32_t scale[32];  // by non-empty event: the largest high word of pt and |m|
  int row[kCapW];      // by row: its particle, and what turns a pair's index into the partner
  uint32_t rows[kRows];  // bit q: a row starts at pair q of the batch
};
static_assert(4 * sizeof(WarpBuf) >= (size_t)kCP * kStagedBytes,
              "an event staged by the CTA takes the place of four warps' buffers");

struct JArgs {
  Lv p;
  const int64_t *off;
  int64_t n_events, n_particles, n_tiles;
  int64_t *pair_off;
  double *pair_m;
  int64_t cap;
  LvOut sums;
  unsigned int *counter;
  unsigned long long *desc;
  int32_t *status;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <int NT, int LP, int LS>
__device__ __noinline__ void big_event(const JArgs &A, int64_t e, int64_t pbeg, int64_t n, int64_t out0) {
  __shared__ double s_red[4 * (NT / 32)];
  // event sum
  double acc[4] = {0, 0, 0, 0};
  for (int64_t k = threadIdx.x; k < n; k += NT) {
    V4<double> v = ld4<double, LP>(A.p, pbeg + k);
    double s, c;
    sincos(v.z, &s, &c);
    Leg<double> l = make_leg(v);
    acc[0] += v.x * c;
    acc[1] += v.x * s;
    acc[2] += v.x * sinh(v.y);
    acc[3] += l.E;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = 0; c < 4; c++) {
    double x = acc[c];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) s_red[c * (NT / 32) + warp] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t[4] = {0, 0, 0, 0};
    for (int c = 0; c < 4; c++)
      for (int w = 0; w < NT / 32; w++) t[c] += s_red[c * (NT / 32) + w];
    st4<double, LS>(A.sums, e, V4<double>{t[0], t[1], t[2], t[3]});
  }
  __syncthreads();
  // pairs, each leg recomputed from global memory
  const int64_t npairs = n * (n - 1) / 2;
  bool over = false;
  for (int64_t k = threadIdx.x; k < npairs; k += NT) {
    int64_t i, j;
    decode_pair_wide(k, n, i, j);
    Leg<double> a = make_leg(ld4<double, LP>(A.p, pbeg + i));
    Leg<double> b = make_leg(ld4<double, LP>(A.p, pbeg + j));
    int64_t dst = out0 + k;
    if (dst < A.cap)
      st_s(A.pair_m + dst, sqrt(pair_terms(a, b).m2));
    else
      over = true;
  }
  if (__syncthreads_or(over) && threadIdx.x == 0) raise_status(A.status, GVX_ERR_CAPACITY);
}

// The Cartesian components of one particle in FP64, out of line (rare).
__device__ __noinline__ void cartesian_f64(V4<double> x, double2 *xy, double2 *ze) {
  double sn, cs;
  sincos(x.z, &sn, &cs);
  *xy = make_double2(x.x * cs, x.x * sn);
  *ze = make_double2(x.x * sinh(x.y), make_leg(x).E);
}

// One particle's terms at its event's scale word wmax, to place c.  False outside the float-float
// domain: then its scale is 0 and, with F64, its FP64 Cartesian components are staged.
template <bool F64>
__device__ __forceinline__ bool stage_particle(const Staged &S, int c, const V4<double> &x,
                                               uint32_t wmax, const ffm::LcTab &T) {
  const double pt = x.x, eta = x.y, phi = x.z, m = x.w;
  const uint32_t hp = ffm::dhi(pt), hm = ffm::dhi(m) & 0x7fffffffu;
  if (ffm::lc_in_domain(hp, hm, ffm::dhi(eta) & 0x7fffffffu, ffm::dhi(phi) & 0x7fffffffu, wmax)) {
    const uint32_t ew = wmax & 0x7ff00000u, rb = ew - (127u << 20);
    const ffm::ff ptf = ffm::cvt1(ffm::cvt_parts(hp, ffm::dlo(pt), rb));
    const ffm::ff mmf = ffm::cvt1(ffm::cvt_parts(hm, ffm::dlo(m), rb));
    const int64_t ae = ffm::angle_fx(eta), ap = ffm::angle_fx(phi);
    uint32_t n, j;
    ffm::ff re = ffm::fx_half_reduce(2 * ae, &n), rp = ffm::fx_half_reduce(2 * ap, &j);
    if (ffm::fx_small(ae, ap)) {  // seldom
      re = ffm::own_reduce(eta, ae, &n);
      rp = ffm::own_reduce(phi, ap, &j);
    }
    ffm::ff sh, sn, cs;
    const ffm::LcLeg<ffm::ff> L = ffm::lc_leg_at(ptf, mmf, re, &n, T.hyp, &sh);
    S.dy[c] = make_float4(L.D.hi, L.Y.hi, L.D.lo, L.Y.lo);
    S.ang[c] = make_longlong2(ae, ap);
    S.pt[c] = make_float2(ptf.hi, ptf.lo);
    S.scale[c] = ew;
    ffm::sincos_lc_at(rp, j, T.sin, &sn, &cs);
    const float sphi = (ffm::dhi(phi) >> 31) ? -1.0f : 1.0f, seta = (ffm::dhi(eta) >> 31) ? -1.0f : 1.0f;
    const ffm::ff px = ffm::lc_mul(ptf, cs), py = ffm::lc_scale(ffm::lc_mul(ptf, sn), sphi);
    const ffm::ff pz = ffm::lc_scale(ffm::lc_mul(ptf, sh), seta);
    S.c0[c] = make_float4(px.hi, py.hi, px.lo, py.lo);
    S.c1[c] = make_float4(pz.hi, L.E.hi, pz.lo, L.E.lo);
    return true;
  }
  if constexpr (F64) cartesian_f64(x, reinterpret_cast<double2 *>(S.c0 + c), reinterpret_cast<double2 *>(S.c1 + c));
  S.scale[c] = 0u;
  return false;
}

// Two components of the sum over places c, c + step, .. < end: float-float terms of the fast-path
// particles in *f (lanes); with F64 also the FP64 terms of the others in d, and the result is the
// event's scale field if any particle is on the fast path (otherwise that of the last particle).
template <bool F64>
__device__ __forceinline__ uint32_t sum_places(const float4 *col, const uint32_t *scale, int c, int end,
                                               int step, ffm::ff2 *f, double *d) {
  ffm::ff2 a = {ffm::bc2(0.0f), ffm::bc2(0.0f)};
  uint32_t ew = 0;
  d[0] = d[1] = 0.0;
  for (; c < end; c += step) {
    const float4 v = col[c];
    const uint32_t w = F64 ? scale[c] : 1u;
    if (w) {
      a = ffm::add_same(a, ffm::ff2{ffm::mk2(v.x, v.y), ffm::mk2(v.z, v.w)});
      ew = w;
    } else {
      const double2 r = *reinterpret_cast<const double2 *>(col + c);
      d[0] += r.x;
      d[1] += r.y;
    }
  }
  if constexpr (!F64) ew = scale[end - 1];
  *f = a;
  return ew;
}

// Components 2 h and 2 h + 1 of event e's sum.
template <int LS>
__device__ __forceinline__ void put_sums(const JArgs &A, int64_t e, int h, double x, double y) {
  if constexpr (LS == GVX_SOA) {
    st_s((double *)(h ? A.sums.c[2] : A.sums.c[0]) + e, x);
    st_s((double *)(h ? A.sums.c[3] : A.sums.c[1]) + e, y);
  } else {
    __stcs((double2 *)A.sums.c[0] + 2 * e + h, make_double2(x, y));
  }
}

__device__ __forceinline__ double sum_to_double(const ffm::ff &f, uint32_t ew, double d) {
  return ew ? ffm::lc_to_double(f, ew - (127u << 20)) + d : d;
}

// One batch by one warp: `take` events of the tile from event sb on (lane l < take having event
// sb + l with particles lo .. hi - 1), together at most kCapW particles.  RARE: a second walk, which
// writes the pairs that the first one left and nothing else.  Returns kOver when a pair did not
// fit the output, kRare when a pair or an event's sums were left.
constexpr int kOver = 1, kRare = 2;

template <int LP, int LS, bool RARE>
__device__ __forceinline__ int warp_batch(const JArgs &A, const ffm::LcTab &T, WarpBuf &W, int64_t e0,
                                          int sb, int take, int64_t lo, int64_t hi, const int64_t *s_pp,
                                          int64_t base) {
  const int lane = threadIdx.x & 31;
  const unsigned upto = 0xffffffffu >> (31 - lane), below = upto >> 1;
  const Staged S = {W.dy, W.ang, W.c0, W.c1, W.pt, W.sc};
  const int64_t pb = __shfl_sync(kAll, lo, 0);
  const int np = (int)(__shfl_sync(kAll, hi, take - 1) - pb);
  const int64_t q0 = s_pp[sb];
  const int total = (int)(s_pp[sb + take] - q0);
  // the particles' loads go out first
  V4<double> x[2];
#pragma unroll
  for (int r = 0; r < 2; r++)
    if (lane + 32 * r < np && GVX_IN_BOUNDS(pb + lane + 32 * r, A.n_particles, A.status))
      x[r] = ld4<double, LP>(A.p, pb + lane + 32 * r);
  // non-empty events in order; the particles they start at as bits
  const int n_l = lane < take ? (int)(hi - lo) : 0, st_l = (int)(lo - pb);
  const unsigned nz = __ballot_sync(kAll, n_l > 0);
  const int nev = __popc(nz);
  const unsigned m0 = __reduce_or_sync(kAll, n_l > 0 && st_l < 32 ? 1u << st_l : 0u);
  const unsigned m1 = __reduce_or_sync(kAll, n_l > 0 && st_l >= 32 ? 1u << (st_l - 32) : 0u);
  if (n_l > 0) {
    const int k = __popc(nz & below);
    W.info[k] = make_int4(st_l, n_l, (int)(s_pp[sb + lane] - q0), sb + lane);
    W.scale[k] = 0u;
  } else if (!RARE && lane < take) {
    put_sums<LS>(A, e0 + sb + lane, 0, 0.0, 0.0);
    put_sums<LS>(A, e0 + sb + lane, 1, 0.0, 0.0);
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
  bool extreme = false;
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const int c = lane + 32 * r;
    if (c < np) {
      const int4 v = W.info[rank[r]];
      const int li = c - v.x;
      if (li + 1 < v.y) {  // a row: pairs first .. first + (n - li - 2), partners c + 1 ..
        const int first = v.z + li * v.y - (li * (li + 1) >> 1);
        W.row[c - rank[r]] = c | (c + 1 - first) << 8;
        atomicOr(&W.rows[first >> 5], 1u << (first & 31));
      }
      extreme |= !stage_particle<RARE>(S, c, x[r], W.scale[rank[r]], T);
    }
  }
  extreme = __any_sync(kAll, extreme);
  __syncwarp();  // the staged places and rows are visible to the warp (a vote orders no memory)
  // event sums: lanes (event, component pair, every other particle); an event with a particle
  // outside the float-float domain gets its sums in the second walk
  if (!RARE || extreme) {
    for (int t = lane; t < 4 * nev; t += 32) {
      const int4 v = W.info[t >> 2];
      const int h = (t >> 1) & 1;
      ffm::ff2 f;
      double d[2];
      uint32_t ew = sum_places<RARE>(h ? S.c1 : S.c0, S.scale, v.x + (t & 1), v.x + v.y, 2, &f, d);
      const unsigned pair = 3u << (lane & 30);
      const ffm::ff2 g = {ffm::mk2(__shfl_xor_sync(pair, f.hi.x, 1), __shfl_xor_sync(pair, f.hi.y, 1)),
                          ffm::mk2(__shfl_xor_sync(pair, f.lo.x, 1), __shfl_xor_sync(pair, f.lo.y, 1))};
      if constexpr (RARE) {
        ew |= __shfl_xor_sync(pair, ew, 1);
        d[0] += __shfl_xor_sync(pair, d[0], 1);
        d[1] += __shfl_xor_sync(pair, d[1], 1);
      }
      if ((t & 1) == 0) {
        f = ffm::add_same(f, g);
        put_sums<LS>(A, e0 + v.w, h, sum_to_double(ffm::lane_x(f), ew, d[0]), sum_to_double(ffm::lane_y(f), ew, d[1]));
      }
    }
  }
  // pairs
  const int64_t dst0 = base + q0, room = A.cap - dst0;
  const int lim = room < total ? (int)(room < 0 ? 0 : room) : total;
  double *const out = A.pair_m + dst0;
  bool rare = false;
  int rows = -1;  // rows that start before the current word, less one
  for (int r0 = 0; r0 < lim; r0 += 32) {
    const unsigned w = W.rows[r0 >> 5];
    const int q = r0 + lane;
    if (q < lim) {
      const int rec = W.row[rows + __popc(w & upto)];
      const int i = rec & 0xff, j = q + (rec >> 8);
      if (GVX_IN_BOUNDS(i, np, A.status) && GVX_IN_BOUNDS(j, np, A.status)) {
        const ffm::EvPart a = S.part(i), b = S.part(j);
        ffm::ff m2s;
        const bool ok = !(extreme && (a.scale == 0u || b.scale == 0u)) && ffm::ev_pair_m2(a, b, T, &m2s);
        if constexpr (RARE) {
          if (!ok) st_s(out + q, pair_mass_at<LP>(A.p.c[0], A.p.c[1], A.p.c[2], A.p.c[3], pb + i, pb + j));
        } else {
          if (ok)
            st_s(out + q, ffm::lc_mass_out(m2s, a.scale));
          else
            rare = true;
        }
      }
    }
    rows += __popc(w);
  }
  __syncwarp();  // before the next batch overwrites the staged particles
  return (lim < total ? kOver : 0) | (rare || extreme ? kRare : 0);
}

// The tile's batches, every warp walking the tile: in the first walk a warp that ends a batch draws the
// number of its next one from *next (their costs differ, and fixed turns leave warps waiting at the
// tile's end: 0.564 ms), in the second they take turns.  *large: an event was left to the CTA.
template <int NT, int LP, int LS, bool RARE>
__device__ __forceinline__ int walk_tile(const JArgs &A, const ffm::LcTab &T, WarpBuf &W, int64_t e0,
                                         int ne, const int64_t *s_off, const int64_t *s_pp, int64_t base,
                                         int *next, bool *large) {
  const int lane = threadIdx.x & 31;
  int seen = 0, mine = threadIdx.x >> 5;
  for (int sb = 0, number = 0; sb < ne; number++) {
    const int64_t lo = s_off[min(sb + lane, ne)], hi = s_off[min(sb + lane + 1, ne)];
    const int64_t pb = __shfl_sync(kAll, lo, 0);
    const int take = __popc(__ballot_sync(kAll, sb + lane < ne && hi - pb <= kCapW));
    if (take == 0) {
      *large = true;
      sb++;
      number--;
      continue;
    }
    if (number == mine) {
      seen |= warp_batch<LP, LS, RARE>(A, T, W, e0, sb, take, lo, hi, s_pp, base);
      if constexpr (RARE) {
        mine += NT / 32;
      } else {
        int t = 0;
        if (lane == 0) t = atomicAdd(next, 1);
        mine = __shfl_sync(kAll, t, 0);
      }
    }
    sb += take;
  }
  return seen;
}

// One event of more than kCapW and at most kCP particles, staged by the whole CTA.
template <int NT, int LP, int LS>
__device__ __forceinline__ bool staged_event(const JArgs &A, const ffm::LcTab &T, const Staged &S, int64_t e,
                                             int64_t pb, int n, int64_t out0) {
  __shared__ uint32_t s_scale;
  if (threadIdx.x == 0) s_scale = 0u;
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += NT) {
    if (!GVX_IN_BOUNDS(pb + c, A.n_particles, A.status)) continue;
    const V4<double> x = ld4c<LP>(A.p, pb + c);
    atomicMax(&s_scale, ffm::umax32(ffm::dhi(x.x), ffm::dhi(x.w) & 0x7fffffffu));
  }
  __syncthreads();
  for (int c = threadIdx.x; c < n; c += NT) {
    if (!GVX_IN_BOUNDS(pb + c, A.n_particles, A.status)) continue;
    stage_particle<true>(S, c, ld4c<LP>(A.p, pb + c), s_scale, T);
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    ffm::ff2 f;
    double d[2];
    const uint32_t ew = sum_places<true>(threadIdx.x ? S.c1 : S.c0, S.scale, 0, n, 1, &f, d);
    put_sums<LS>(A, e, threadIdx.x, sum_to_double(ffm::lane_x(f), ew, d[0]), sum_to_double(ffm::lane_y(f), ew, d[1]));
  }
  const int total = n * (n - 1) / 2;
  bool fits = true;
  for (int q = threadIdx.x; q < total; q += NT) {
    int i, j;
    decode_pair32(q, n, i, j);
    if (!(GVX_IN_BOUNDS(i, n, A.status) && GVX_IN_BOUNDS(j, n, A.status))) continue;
    if (out0 + q >= A.cap) {
      fits = false;
      continue;
    }
    const ffm::EvPart a = S.part(i), b = S.part(j);
    ffm::ff m2s;
    if (a.scale != 0u && b.scale != 0u && ffm::ev_pair_m2(a, b, T, &m2s))
      st_s(A.pair_m + out0 + q, ffm::lc_mass_out(m2s, a.scale));
    else
      st_s(A.pair_m + out0 + q, pair_mass_at<LP>(A.p.c[0], A.p.c[1], A.p.c[2], A.p.c[3], pb + i, pb + j));
  }
  __syncthreads();
  return fits;
}

// What the batches of a tile left, by the whole CTA.
template <int NT, int LP, int LS>
__device__ __noinline__ void finish_tile(const JArgs &A, unsigned char *s_dyn, int64_t e0, int ne,
                                         const int64_t *s_off, const int64_t *s_pp, int64_t base, bool rare) {
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};
  bool large;
  if (rare)
    walk_tile<NT, LP, LS, true>(A, T, reinterpret_cast<WarpBuf *>(s_dyn)[threadIdx.x >> 5], e0, ne, s_off, s_pp,
                                base, nullptr, &large);
  __syncthreads();
  Staged S;
  S.dy = reinterpret_cast<float4 *>(s_dyn);
  S.ang = reinterpret_cast<longlong2 *>(S.dy + kCP);
  S.c0 = reinterpret_cast<float4 *>(S.ang + kCP);
  S.c1 = S.c0 + kCP;
  S.pt = reinterpret_cast<float2 *>(S.c1 + kCP);
  S.scale = reinterpret_cast<uint32_t *>(S.pt + kCP);
  for (int e = 0; e < ne; e++) {
    const int64_t pb = s_off[e], n = s_off[e + 1] - pb;
    if (n <= kCapW) continue;
    bool fits = true;
    if (n <= kCP)
      fits = staged_event<NT, LP, LS>(A, T, S, e0 + e, pb, (int)n, base + s_pp[e]);
    else
      big_event<NT, LP, LS>(A, e0 + e, pb, n, base + s_pp[e]);
    if (!fits) raise_status(A.status, GVX_ERR_CAPACITY);
  }
  __syncthreads();
}

// The pairs before tile `tile`, by one warp: its own total published first, then the descriptors
// before it read 32 at a time, back to the nearest inclusive prefix.
__device__ __forceinline__ int64_t look_back(const JArgs &A, int64_t tile, int64_t tile_total) {
  const int lane = threadIdx.x & 31;
  int64_t prefix = 0;
  if (tile > 0) {
    if (lane == 0) st_relaxed(&A.desc[tile], kFlagAgg | (unsigned long long)tile_total);
    unsigned long long t0 = 0, polls = 0;
    for (int64_t j = tile - 1; j >= 0;) {
      // lane l: descriptor j - l; before the first tile there is an inclusive prefix of 0
      const unsigned long long d = j - lane >= 0 ? ld_relaxed(&A.desc[j - lane]) : kFlagInc;
      const unsigned long long f = d & ~kValMask;
      const unsigned inc = __ballot_sync(kAll, f == kFlagInc), none = __ballot_sync(kAll, f == 0);
      const int last = inc ? __ffs((int)inc) - 1 : 31;  // the words up to `last` are needed
      if (none & (0xffffffffu >> (31 - last))) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        const bool give_up = now - t0 > kWaitLimitNs || ++polls > kMaxPolls;
        if (__any_sync(kAll, give_up)) {
          if (lane == 0) raise_status(A.status, GVX_ERR_TIMEOUT);
          break;
        }
        __nanosleep(64);
        continue;
      }
      int64_t v = lane <= last ? (int64_t)(d & kValMask) : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
      prefix += v;
      if (inc) break;
      j -= 32;
    }
  }
  if (lane == 0) st_relaxed(&A.desc[tile], kFlagInc | (unsigned long long)(prefix + tile_total));
  return prefix;
}

template <int TE, int NT, int LP, int LS>
__global__ void __launch_bounds__(NT, 768 / NT) event_pairs_kernel(const __grid_constant__ JArgs A) {
  static_assert(TE <= NT && NT % 128 == 0, "one event per thread in the tile scan");
  extern __shared__ __align__(16) unsigned char s_dyn[];
  WarpBuf *bufs = reinterpret_cast<WarpBuf *>(s_dyn);
  __shared__ int64_t s_off[TE + 1];
  __shared__ int64_t s_pp[TE + 1];
  __shared__ int64_t s_warp[NT / 32];
  __shared__ int64_t s_base;
  __shared__ int64_t s_tile;
  __shared__ int s_next;
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  for (;;) {
    if (threadIdx.x == 0) {
      s_tile = (int64_t)atomicAdd(A.counter, 1u);
      s_next = NT / 32;
    }
    __syncthreads();
    const int64_t tile = s_tile;
    if (tile >= A.n_tiles) break;
    const int64_t e0 = tile * TE;
    const int ne = (int)((A.n_events - e0) < TE ? (A.n_events - e0) : TE);

    // 1. offsets, validation, pair counts, tile scan
    for (int k = threadIdx.x; k <= ne; k += NT) s_off[k] = A.off[e0 + k];
    __syncthreads();
    bool bad = false;
    if (threadIdx.x < ne) {
      int64_t lo = s_off[threadIdx.x], hi = s_off[threadIdx.x + 1];
      bad = lo < 0 || hi < lo || hi > A.n_particles;
    }
    if (threadIdx.x == 0) {
      if (tile == 0 && s_off[0] != 0) bad = true;
      if (tile == A.n_tiles - 1 && s_off[ne] != A.n_particles) bad = true;
    }
    const bool tile_bad = __syncthreads_or(bad);
    if (tile_bad) {  // treat every event of the tile as empty: nothing is read or written
      if (threadIdx.x == 0) raise_status(A.status, GVX_ERR_OFFSETS);
      __syncthreads();
      for (int k = threadIdx.x; k <= ne; k += NT) s_off[k] = 0;
      __syncthreads();
    }
    int64_t cnt = threadIdx.x < ne ? s_off[threadIdx.x + 1] - s_off[threadIdx.x] : 0;
    int64_t tile_total;
    int64_t excl = block_excl_scan<NT>(cnt * (cnt - 1) / 2, s_warp, &tile_total);
    if (threadIdx.x < ne) s_pp[threadIdx.x] = excl;
    if (threadIdx.x == 0) s_pp[ne] = tile_total;

    // 2. decoupled look-back
    if (warp == 0) {
      const int64_t prefix = look_back(A, tile, tile_total);
      if (lane == 0) s_base = prefix;
    }
    __syncthreads();
    const int64_t base = s_base;
    if (threadIdx.x < ne) A.pair_off[e0 + threadIdx.x] = base + s_pp[threadIdx.x];
    if (tile == A.n_tiles - 1 && threadIdx.x == 0) A.pair_off[A.n_events] = base + tile_total;

    // 3. the batches, 4. what they leave
    bool large = false;
    const int seen = walk_tile<NT, LP, LS, false>(A, T, bufs[warp], e0, ne, s_off, s_pp, base, &s_next,
                                                        &large);
    if ((seen & kOver) && lane == 0) raise_status(A.status, GVX_ERR_CAPACITY);
    const bool rare = __syncthreads_or(seen & kRare);
    if (rare || large) finish_tile<NT, LP, LS>(A, s_dyn, e0, ne, s_off, s_pp, base, rare);
  }
}

// Tile shapes the autotuner chooses among: (events per tile, threads per CTA).
struct Shape {
  int te, nt;
};
constexpr Shape kShapes[] = {{64, 128}, {128, 128}, {128, 256}, {256, 256}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);

template <int TE, int NT, int LP, int LS>
cudaError_t launch_shape(const JArgs &A0, bool skip_first_tile, cudaStream_t s) {
  auto kern = event_pairs_kernel<TE, NT, LP, LS>;
  constexpr size_t kDynSmem = (NT / 32) * sizeof(WarpBuf);
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kDynSmem);
  if (err != cudaSuccess) return err;
  int per_sm = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, kDynSmem);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) per_sm = 1;
  JArgs A = A0;
  A.n_tiles = (A.n_events + TE - 1) / TE;
  int64_t grid = (int64_t)num_sms() * per_sm;
  if (grid > A.n_tiles) grid = A.n_tiles;
  if (grid < 1) grid = 1;
  // tile counter + one descriptor per tile start at zero
  err = cudaMemsetAsync(A.counter, 0, kWsHeader + (size_t)A.n_tiles * 8, s);
  if (err != cudaSuccess) return err;
  if (skip_first_tile) {  // test hook: tile 0 is never taken, so its successors' waits time out
    err = cudaMemsetAsync(A.counter, 1, 1, s);
    if (err != cudaSuccess) return err;
  }
  kern<<<(unsigned)grid, NT, kDynSmem, s>>>(A);
  return cudaGetLastError();
}

template <int LP, int LS>
cudaError_t launch_any_shape(int shape, const JArgs &A, bool skip, cudaStream_t s) {
  switch (shape) {
    case 0: return launch_shape<64, 128, LP, LS>(A, skip, s);
    case 1: return launch_shape<128, 128, LP, LS>(A, skip, s);
    case 2: return launch_shape<128, 256, LP, LS>(A, skip, s);
    default: return launch_shape<256, 256, LP, LS>(A, skip, s);
  }
}

}  // namespace

int event_pairs_num_shapes() { return kNumShapes; }

void event_pairs_shape(int shape, int *te, int *nt) {
  if (shape < 0 || shape >= kNumShapes) shape = 0;
  *te = kShapes[shape].te;
  *nt = kShapes[shape].nt;
}

size_t event_pairs_workspace(int64_t n_events) {
  return kWsHeader + (size_t)((n_events + kMinTE - 1) / kMinTE) * 8;
}

cudaError_t launch_event_pairs_shape(int shape, const Lv &p, const int64_t *off, int64_t n_events,
                                     int64_t n_particles, int64_t *pair_off, double *pair_m,
                                     int64_t capacity, const LvOut &sums, void *ws,
                                     bool skip_first_tile, cudaStream_t s) {
  JArgs A;
  A.p = p;
  A.off = off;
  A.n_events = n_events;
  A.n_particles = n_particles;
  A.n_tiles = 0;
  A.pair_off = pair_off;
  A.pair_m = pair_m;
  A.cap = capacity;
  A.sums = sums;
  A.counter = (unsigned int *)ws;
  A.desc = (unsigned long long *)((char *)ws + kWsHeader);
  A.status = device_status_word();
  if (!A.status) return cudaErrorInvalidSymbol;
  const bool k = skip_first_tile;
  if (p.layout == GVX_SOA && sums.layout == GVX_SOA)
    return launch_any_shape<GVX_SOA, GVX_SOA>(shape, A, k, s);
  if (p.layout == GVX_SOA) return launch_any_shape<GVX_SOA, GVX_AOS>(shape, A, k, s);
  if (sums.layout == GVX_SOA) return launch_any_shape<GVX_AOS, GVX_SOA>(shape, A, k, s);
  return launch_any_shape<GVX_AOS, GVX_AOS>(shape, A, k, s);
}

}  // namespace gvx
