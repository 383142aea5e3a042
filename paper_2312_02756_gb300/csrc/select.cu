// Fused per-event analysis step: particle selection, a histogram of the pair masses of the
// selected particles, and per event the selected pair whose mass is closest to a target (the
// RDataFrame-style use of the per-event combinatorics that GenVectorX names as its next target,
// Sec. 6; the pair mass is that of Sec. 4.1, Fig. 1).  No pair mass is written to memory.
//
// Each warp takes tiles of up to 32 consecutive events (one per lane) and works through them in
// batches of its own, synchronised within the warp alone:
//   (a) batches of whole events of at most kRaw particles: the cuts, one ballot per 32 particles;
//   (b) of those, runs of whole events with at most kCap selected particles: each selected particle's
//       raw values go to its place in a compacted list (the place from the ballots), each event
//       finds its scale (the largest high word of pt and |m| over its selected particles) and its
//       number of selected pairs, and the list is turned into light-cone terms with fixed-point
//       angles (event_lc.cuh), 32 at a time;
//   (c) the selected pairs of the run, 32 at a time: the pair mass, its histogram slot (shared-memory
//       integer atomics, so the totals do not depend on the order) and its |m - target|, of which
//       each event keeps the first smallest: the leading words by an integer atomic minimum, the
//       pairs that reach it (one, but for near ties) by their exact (|m - target|, k) -- exact, and
//       the smaller packed index k (the order of gvx_event_pair_masses) on ties.
// What the tiles leave is done after all of a CTA's tiles, in a function of its own (a call inside
// the tiles costs them spills): pairs outside the float-float domain (near-equal directions, extreme
// particles), by walking their tiles once more with the elementwise arithmetic for those pairs, and
// events of more than kCap particles, by the whole block: staged up to kNT particles, else every
// pair from global memory.  At the end each CTA adds its histogram to the caller's counts.
//
// Bound by instruction issue and the latency of its loads (32 M warp instructions at 2^18 events;
// HBM reads 5% of the time).  2^20 events, 4.2 M selected pairs: 0.188 ms a call, against 0.736 ms
// for CTA-wide batches of 256 particles, where ten warps in eleven waited at a block barrier; the
// warps' own batches have none.  Three CTAs of 256 threads per SM: two (0.214 ms) leave too few
// warps for the load latency, four (64 registers, 0.201 ms) spill and crowd the tables out of L1.
#include <cuda_runtime.h>

#include <math.h>

#include "common.cuh"
#include "event_lc.cuh"
#include "pair_index.cuh"
#include "pair_raw.cuh"
#include "select_cuts.cuh"

namespace gvx {
namespace {

constexpr int kNT = 256;      // threads per CTA, and particles of an event the block stages
constexpr int kWarps = kNT / 32;
constexpr int kRaw = 256;     // particles per batch of a warp (eight ballots)
constexpr int kCap = 128;     // selected particles per run, and particles of an event a warp takes
constexpr int kMaxTile = 32;  // events per warp tile, at most
constexpr unsigned kAll = 0xffffffffu;
// A slot of the CTA's histogram has 32 bits.  At most it takes, between two flushes, the pairs of
// kMaxTurns tiles of each warp in either walk (the grid is large enough for that), of staged events up to
// kFlushPairs (and one event more), and of one part of a larger event.
constexpr int kMaxTurns = 256;
constexpr long long kFlushPairs = 1ll << 30;
static_assert(kFlushPairs % kNT == 0 &&
                  2ll * kWarps * kMaxTurns * kMaxTile * (kCap * (kCap - 1) / 2) + 2 * kFlushPairs +
                          kNT * (kNT - 1) / 2 < (1ll << 32),
              "no slot can wrap around");

struct SArgs {
  Lv p;
  const int64_t *off;
  int64_t n_events, n_particles;
  Cuts cuts;
  double lo, hi, inv_w, target;
  float lo_h, lo_l, inv_f, tol0;  // the float histogram slot (slot_of_ff)
  int n_bins, tile, turns;        // tile: events per warp tile; turns: a warp's tiles per bit of its rare mask
  unsigned long long *counts;
  int64_t *best_k;
  double *best_m;
  int32_t *status;
};

// One warp's part of shared memory.
struct __align__(16) WarpBuf {
  ffm::EvPart part[kCap];        // by compacted place; tag: position in the batch | event << 8
  // by event (lane) of the tile: the best pair so far -- the leading word and the bits of its
  // |m - target|, its mass, its particles' positions in the batch (-1: none)
  unsigned long long bd[32];
  double bm[32];
  uint32_t key[32];
  int bk[32], own[32];
  int pp[32], cs[32], n[32];     // by event: first pair and place in the run, selected particles
  uint32_t scale[32];            // by event: the largest high word of pt and |m|
};

// Offsets lo, hi of event e that cannot be right.
__device__ __forceinline__ bool bad_event(const SArgs &A, int64_t e, int64_t lo, int64_t hi) {
  return lo < 0 || hi < lo || hi > A.n_particles || (e == 0 && lo != 0) ||
         (e == A.n_events - 1 && hi != A.n_particles);
}

// The CTA's histogram moved to the caller's counts, by the whole block with no warp counting meanwhile.
__device__ __forceinline__ void flush_slots(const SArgs &A, unsigned *s_hist) {
  for (int s = threadIdx.x; s < A.n_bins + 2; s += kNT) {
    if (s_hist[s]) atomicAdd(A.counts + s, (unsigned long long)s_hist[s]);
    s_hist[s] = 0u;
  }
}

// Histogram slot of a mass: 0 below lo, n_bins + 1 at or above hi (and NaN), else 1 + the bin
// floor((m - lo) * inv_w) clamped to the range (both operations rounded as written).
__device__ __forceinline__ int slot_of(double m, const SArgs &A) {
  if (m < A.lo) return 0;
  if (!(m < A.hi)) return A.n_bins + 1;
  long long b = __double2ll_rz(__dmul_rn(__dsub_rn(m, A.lo), A.inv_w));
  b = b < 0 ? 0 : b;
  b = b > A.n_bins - 1 ? A.n_bins - 1 : b;
  return (int)b + 1;
}

// The same slot from the mass in float-float at scale 2^(sf's exponent), or -1 where floats do not
// decide it: t = (m - lo) inv_w is within tol of its exact value (three roundings of 2^-24 of t,
// and 2^-40 of the range for the low parts left out), so its floor is the bin unless t is within
// tol of an integer.  The FP64 slot costs six operations of a pipe that a warp instruction holds
// for ~77 cycles; about one pair in 10^4 needs it (200 bins).
__device__ __forceinline__ int slot_of_ff(ffm::ff m, float sf, const SArgs &A) {
  const float x = __fadd_rn(__fsub_rn(__fmul_rn(m.hi, sf), A.lo_h), __fsub_rn(__fmul_rn(m.lo, sf), A.lo_l));
  float t = __fmul_rn(x, A.inv_f);
  t = fminf(fmaxf(t, -0.5f), (float)A.n_bins + 0.5f);
  const float tol = __fmaf_rn(fabsf(t), 4.76837158e-07f, A.tol0);  // 2^-21
  return fabsf(t - rintf(t)) > tol ? (int)floorf(t) + 1 : -1;
}

// (d, k) before (d', k'): the smaller |m - target|, NaN last, then the smaller k; k < 0 is "none".  (NaN
// last, because a thread's first pair may have none while its later ones do.)
__device__ __forceinline__ bool better(double d, long long k, double d0, long long k0) {
  return k >= 0 && (k0 < 0 || d < d0 || (d == d0 && k < k0) || (isnan(d0) && (!isnan(d) || k < k0)));
}

// pt and eta of one particle.
template <int LP>
__device__ __forceinline__ void ld_pt_eta(const Lv &v, int64_t i, double &pt, double &eta) {
  if constexpr (LP == GVX_SOA) {
    pt = __ldg((const double *)v.c[0] + i);
    eta = __ldg((const double *)v.c[1] + i);
  } else {
    const double2 a = __ldg((const double2 *)v.c[0] + 2 * i);
    pt = a.x;
    eta = a.y;
  }
}

// A selected particle's place until the leg phase: its raw values (pt, m, eta, phi) and its tag.
__device__ __forceinline__ void stage_raw(ffm::EvPart &P, const V4<double> &x, uint32_t tag) {
  *reinterpret_cast<double2 *>(&P.dy) = make_double2(x.x, x.w);
  *reinterpret_cast<double2 *>(&P.eta) = make_double2(x.y, x.z);
  P.tag = tag;
}

// The place from its raw values to light-cone terms at its event's scale word; false outside the
// float-float domain.
__device__ __forceinline__ bool stage_leg(ffm::EvPart &P, uint32_t wmax, const ffm::LcTab &T) {
  const double2 a = *reinterpret_cast<const double2 *>(&P.dy);
  const double2 b = *reinterpret_cast<const double2 *>(&P.eta);
  const double pt = a.x, m = a.y, eta = b.x, phi = b.y;
  const uint32_t hp = ffm::dhi(pt), hm = ffm::dhi(m) & 0x7fffffffu;
  if (!ffm::lc_in_domain(hp, hm, ffm::dhi(eta) & 0x7fffffffu, ffm::dhi(phi) & 0x7fffffffu, wmax)) {
    P.scale = 0u;
    return false;
  }
  const uint32_t ew = wmax & 0x7ff00000u, rb = ew - (127u << 20);
  const ffm::ff ptf = ffm::cvt1(ffm::cvt_parts(hp, ffm::dlo(pt), rb));
  const ffm::ff mmf = ffm::cvt1(ffm::cvt_parts(hm, ffm::dlo(m), rb));
  const int64_t ae = ffm::angle_fx(eta);
  uint32_t n;
  const ffm::ff r = ffm::fx_half_reduce(2 * ae, &n);
  const ffm::LcLeg<ffm::ff> L = ffm::lc_leg_at(ptf, mmf, r, &n, T.hyp);
  P = ffm::EvPart{make_float4(L.D.hi, L.Y.hi, L.D.lo, L.Y.lo), ae, ffm::angle_fx(phi), ptf.hi, ptf.lo, ew, P.tag};
  return true;
}

// A pair's mass from its scaled m^2 at the scale field ew; with COUNT its histogram slot counted.
template <bool COUNT>
__device__ __forceinline__ double mass_of(ffm::ff m2s, uint32_t ew, const SArgs &A, unsigned *s_hist) {
  ffm::ff r = {0.0f, 0.0f};
  double m = 0.0;
  if (m2s.hi != 0.0f) {
    r = ffm::lc_sqrt_refined(m2s);
    r = ffm::fast_two_sum(r.hi, r.lo);
    m = ffm::lc_to_double_int(r, ew - (127u << 20));
  }
  if constexpr (!COUNT) return m;
  int slot = -1;
  // 2^(scale) as a float where it is one (2^-100 .. 2^100)
  if (ew - (923u << 20) <= (200u << 20)) slot = slot_of_ff(r, __uint_as_float((ew - (896u << 20)) << 3), A);
  if (slot < 0) slot = slot_of(m, A);
  atomicAdd(&s_hist[slot], 1u);
  return m;
}

// One event of more than kNT particles, by the whole block from global memory.
template <int LP>
__device__ __noinline__ void big_event_select(const SArgs &A, const ffm::LcTab &T, unsigned *s_hist, int64_t pb,
                                 int64_t n, double *bd_out, long long *bk_out, double *bm_out) {
  double bd = INFINITY, bm = NAN;
  long long bk = -1;
  const long long npairs = (long long)n * (n - 1) / 2;
  for (long long k0 = 0; k0 < npairs; k0 += kFlushPairs) {
    const long long k1 = npairs - k0 < kFlushPairs ? npairs : k0 + kFlushPairs;
    for (long long k = k0 + threadIdx.x; k < k1; k += kNT) {
      int64_t i, j;
      decode_pair_wide(k, n, i, j);
      const V4<double> x = ld4c<LP>(A.p, pb + i), y = ld4c<LP>(A.p, pb + j);
      if (!(passes(x.x, x.y, A.cuts) && passes(y.x, y.y, A.cuts))) continue;
      const double m = pair_mass_raw(x, y, T);
      atomicAdd(&s_hist[slot_of(m, A)], 1u);
      const double d = fabs(m - A.target);
      if (better(d, k, bd, bk)) {
        bd = d;
        bk = k;
        bm = m;
      }
    }
    __syncthreads();  // all of these counted before any of the next
    flush_slots(A, s_hist);
    __syncthreads();
  }
  *bd_out = bd;
  *bk_out = bk;
  *bm_out = bm;
}

// One event of more than kCap and at most kNT particles, staged by the whole block: a particle per
// thread, then its selected pairs over all threads.
template <int LP>
__device__ __noinline__ void staged_event_select(const SArgs &A, const ffm::LcTab &T, ffm::EvPart *part,
                                                 unsigned *s_hist, int64_t pb, int n, double *bd_out,
                                                 long long *bk_out, double *bm_out) {
  __shared__ int64_t s_warp[kWarps];
  __shared__ unsigned s_scale;
  const int k = threadIdx.x;
  V4<double> x = {0.0, 0.0, 0.0, 0.0};
  const bool in = k < n;
  if (in) x = ld4<double, LP>(A.p, pb + k);
  const bool pass = in && passes(x.x, x.y, A.cuts);
  if (k == 0) s_scale = 0u;
  int64_t nsel;
  const int c = (int)block_excl_scan<kNT>(pass ? 1 : 0, s_warp, &nsel);  // ends synchronised
  if (pass) {
    stage_raw(part[c], x, (uint32_t)k);
    atomicMax(&s_scale, ffm::umax32(ffm::dhi(x.x), ffm::dhi(x.w) & 0x7fffffffu));
  }
  __syncthreads();
  if (k < (int)nsel) stage_leg(part[k], s_scale, T);
  __syncthreads();
  const int ns = (int)nsel, total = ns * (ns - 1) / 2;
  double bd = INFINITY, bm = NAN;
  long long bk = -1;
  for (int q = k; q < total; q += kNT) {
    int i, j;
    decode_pair32(q, ns, i, j);
    const ffm::EvPart &a = part[i], &b = part[j];
    const int oi = (int)a.tag, oj = (int)b.tag;
    ffm::ff m2s;
    double m;
    if (a.scale != 0u && b.scale != 0u && ffm::ev_pair_m2(a, b, T, &m2s)) {
      m = mass_of<true>(m2s, a.scale, A, s_hist);
    } else {
      m = pair_mass_at<LP>(A.p.c[0], A.p.c[1], A.p.c[2], A.p.c[3], pb + oi, pb + oj);
      atomicAdd(&s_hist[slot_of(m, A)], 1u);
    }
    double d = fabs(m - A.target);
    if (q == 0 && isnan(d)) d = -1.0;  // a first pair without a distance is never replaced
    const long long kk = oi * n - oi * (oi + 1) / 2 + (oj - oi - 1);
    if (better(d, kk, bd, bk)) {
      bd = d;
      bk = kk;
      bm = m;
    }
  }
  *bd_out = bd;
  *bk_out = bk;
  *bm_out = bm;
}

// The particles of pair q of a run: places ci, cj and the event (lane) e.
__device__ __forceinline__ void pair_places(const WarpBuf &W, int q, int &e, int &ci, int &cj) {
  e = 0;  // the last event whose first pair is <= q
#pragma unroll
  for (int step = 16; step > 0; step >>= 1)
    if (W.pp[e + step] <= q) e += step;
  int i, j;
  decode_pair32(q - W.pp[e], W.n[e], i, j);
  ci = W.cs[e] + i;
  cj = W.cs[e] + j;
}

// Pairs of mass m and particle positions k (row-major order as an integer) offered to their events'
// best, by the whole warp; first: the event's first pair, which stays if it has no distance (NaN).
__device__ __forceinline__ void offer(WarpBuf &W, bool valid, int e, double m, int k, bool first,
                                      const SArgs &A) {
  const int lane = threadIdx.x & 31;
  // distances are non-negative: their bits order them, NaN last
  unsigned long long d = (unsigned long long)__double_as_longlong(fabs(m - A.target));
  if (first && d > 0x7ff0000000000000ull) d = 0ull;
  const uint32_t key = (uint32_t)(d >> 32);
  if (valid) atomicMin(&W.key[e], key);
  __syncwarp();
  bool cand = valid && key == W.key[e];
  __syncwarp();  // every lane has read its key before the next round lowers one
  while (__any_sync(kAll, cand)) {
    if (cand) W.own[e] = lane;
    __syncwarp();
    if (cand && W.own[e] == lane) {
      const unsigned long long d0 = W.bd[e];
      const int k0 = W.bk[e];
      if (k0 < 0 || d < d0 || (d == d0 && k < k0)) {
        W.bd[e] = d;
        W.bm[e] = m;
        W.bk[e] = k;
      }
      cand = false;
    }
    __syncwarp();
  }
}

// One warp tile: events e0 .. e0 + ne - 1 (ne <= 32), lane l having event e0 + l with particles
// lo .. hi - 1.  Returns kLarge when it left an event to the block, kRare when it left a pair to a
// second walk.  RARE: that walk, which counts the pairs left and forms the best ones anew.
constexpr int kLarge = 1, kRare = 2;

template <int LP, bool RARE>
__device__ __forceinline__ int warp_tile(const SArgs &A, const ffm::LcTab &T, WarpBuf &W,
                                          unsigned *s_hist, int64_t e0, int ne, int64_t lo, int64_t hi) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  W.key[lane] = 0xffffffffu;
  W.bk[lane] = -1;
  W.bm[lane] = NAN;
  int left = 0;
  if (__any_sync(kAll, lane < ne && bad_event(A, e0 + lane, lo, hi))) {
    // nothing of the tile is read; its events report no candidate
    if (lane == 0) raise_status(A.status, GVX_ERR_OFFSETS);
  } else {
    int sb = 0;
    while (sb < ne) {
      // (a) a batch of whole events: at most kRaw particles, none of more than kCap
      const int64_t pb = __shfl_sync(kAll, lo, sb);
      const unsigned ok =
          __ballot_sync(kAll, lane >= sb && lane < ne && hi - lo <= kCap && hi - pb <= kRaw) >> sb;
      const int take = ok == kAll ? 32 : __ffs((int)~ok) - 1;  // the leading ones that fit
      if (take == 0) {  // an event for the block
        left |= kLarge;
        sb++;
        continue;
      }
      const int sbe = sb + take;
      const int np = (int)(__shfl_sync(kAll, hi, sbe - 1) - pb);
      unsigned word = 0;  // lane r: the selection bits of particles 32 r .. 32 r + 31
      for (int r = 0; r < np; r += 128) {
        double pt[4], eta[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          pt[u] = eta[u] = NAN;  // fails the cuts
          if (r + 32 * u + lane < np) ld_pt_eta<LP>(A.p, pb + r + 32 * u + lane, pt[u], eta[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const unsigned b = __ballot_sync(kAll, passes(pt[u], eta[u], A.cuts));
          if (lane == r / 32 + u) word = b;
        }
      }
      // selected particles before position 32 lane, then before each event's first particle and
      // before the one after its last
      int pre = __popc(word);
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const int y = __shfl_up_sync(kAll, pre, o);
        if (lane >= o) pre += y;
      }
      pre -= __popc(word);
      const bool mine = lane >= sb && lane < sbe;
      const int s0 = mine ? (int)(lo - pb) : np, s1 = mine ? (int)(hi - pb) : np;
      const int w0 = __shfl_sync(kAll, (int)word, s0 >> 5), f0 = __shfl_sync(kAll, pre, s0 >> 5);
      const int w1 = __shfl_sync(kAll, (int)word, s1 >> 5), f1 = __shfl_sync(kAll, pre, s1 >> 5);
      const int c0 = f0 + __popc((unsigned)w0 & ((1u << (s0 & 31)) - 1u));
      const int c1 = f1 + __popc((unsigned)w1 & ((1u << (s1 & 31)) - 1u));
      // (b), (c) runs of whole events with at most kCap selected particles
      int rb = sb;
      while (rb < sbe) {
        const int cbase = __shfl_sync(kAll, c0, rb);
        const int re = rb + __popc(__ballot_sync(kAll, lane >= rb && lane < sbe && c1 - cbase <= kCap));
        const int ns = __shfl_sync(kAll, c1, re - 1) - cbase;  // re > rb: an event has at most kCap
        const bool run = lane >= rb && lane < re;
        const int nse = run ? c1 - c0 : 0;
        int pp = nse * (nse - 1) / 2;
        const int npairs = pp;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kAll, pp, o);
          if (lane >= o) pp += y;
        }
        const int total = __shfl_sync(kAll, pp, 31);
        if (total > 0) {
          W.pp[lane] = pp - npairs;
          W.cs[lane] = c0 - cbase;
          W.n[lane] = nse;
          // the selected particles of the run, each at its place
          const int first = (int)(__shfl_sync(kAll, lo, rb) - pb);
          const int last = (int)(__shfl_sync(kAll, hi, re - 1) - pb);
          for (int r = first & ~31; r < last; r += 32) {
            const unsigned b = (unsigned)__shfl_sync(kAll, (int)word, r >> 5);
            const int f = __shfl_sync(kAll, pre, r >> 5) - cbase;
            const int i = r + lane;
            if (((b >> lane) & 1u) && i >= first && i < last) {
              stage_raw(W.part[f + __popc(b & below)], ld4c<LP>(A.p, pb + i), (uint32_t)i);
            }
          }
          __syncwarp();
          if (run) {  // the event's scale; its particles learn their event
            uint32_t wmax = 0;
            for (int c = c0 - cbase; c < c1 - cbase; c++) {
              const double2 a = *reinterpret_cast<const double2 *>(&W.part[c].dy);
              wmax = ffm::umax32(ffm::umax32(ffm::dhi(a.x), ffm::dhi(a.y) & 0x7fffffffu), wmax);
              W.part[c].tag |= (uint32_t)lane << 8;
            }
            W.scale[lane] = wmax;
          }
          __syncwarp();
          bool extreme = false;
          for (int c = lane; c < ns; c += 32)
            extreme |= !stage_leg(W.part[c], W.scale[W.part[c].tag >> 8], T);
          extreme = __any_sync(kAll, extreme);
          __syncwarp();  // the staged places are visible to the warp (a vote orders no memory)
          bool rare = false;
          for (int r0 = 0; r0 < total; r0 += 32) {
            const int q = r0 + lane;
            int e = 0, k = 0;
            bool offered = false, fst = false;
            double m = 0.0;
            if (q < total) {
              int ci, cj;
              pair_places(W, q, e, ci, cj);
              const ffm::EvPart &a = W.part[ci], &b = W.part[cj];
              const int oi = a.tag & 0xff, oj = b.tag & 0xff;
              ffm::ff m2s;
              const bool fast = !(extreme && (a.scale == 0u || b.scale == 0u)) && ffm::ev_pair_m2(a, b, T, &m2s);
              if (fast) m = mass_of<!RARE>(m2s, a.scale, A, s_hist);
              if constexpr (RARE) {
                if (!fast) {
                  m = pair_mass_at<LP>(A.p.c[0], A.p.c[1], A.p.c[2], A.p.c[3], pb + oi, pb + oj);
                  atomicAdd(&s_hist[slot_of(m, A)], 1u);
                }
              }
              offered = RARE || fast;
              rare |= !fast;
              k = oi << 8 | oj;
              fst = q == W.pp[e];
            }
            offer(W, offered, e, m, k, fst, A);
          }
          if (__any_sync(kAll, rare)) left |= kRare;
          __syncwarp();  // before the next run's particles
          if (run && W.bk[lane] >= 0) {  // positions in the batch -> the packed index in the event
            const int n = (int)(hi - lo), k = W.bk[lane];
            const int i = (k >> 8) - (int)(lo - pb), j = (k & 0xff) - (int)(lo - pb);
            W.bk[lane] = i * n - i * (i + 1) / 2 + (j - i - 1);
          }
        }
        rb = re;
      }
      sb = sbe;
    }
  }
  __syncwarp();
  if (lane < ne) {
    if (A.best_k) A.best_k[e0 + lane] = W.bk[lane];
    if (A.best_m) A.best_m[e0 + lane] = W.bm[lane];
  }
  __syncwarp();
  return left;
}

// Asks L2 for the lines of particles lo .. hi - 1 (nothing for a range that cannot be right).
template <int LP>
__device__ __forceinline__ void prefetch_particles(const SArgs &A, int64_t lo, int64_t hi) {
  if (lo < 0 || hi <= lo || hi > A.n_particles || hi - lo > 1024) return;
  const int bytes = (int)(hi - lo) * (LP == GVX_SOA ? 8 : 32);
#pragma unroll
  for (int c = 0; c < (LP == GVX_SOA ? 4 : 1); c++) {
    const char *p = (const char *)A.p.c[c] + lo * (LP == GVX_SOA ? 8 : 32);
    for (int o = 128 * (threadIdx.x & 31); o < bytes; o += 128 * 32)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
  }
}

// Events of warp tile t.
__device__ __forceinline__ int events_of(const SArgs &A, int64_t t) {
  const int64_t rest = A.n_events - t * A.tile;
  return (int)(rest < A.tile ? rest : A.tile);
}

// What the tiles of a CTA left: rare, per warp, the tiles with pairs to walk again; then the events
// of more than kCap particles, by the whole block.
template <int LP>
__device__ __noinline__ void finish_tiles(const SArgs &A, unsigned char *s_dyn, unsigned *s_hist,
                                          int64_t n_tiles, unsigned long long rare) {
  __shared__ int64_t s_off[kWarps][kMaxTile + 1];
  __shared__ int s_ne[kWarps];
  __shared__ double s_rd[kNT], s_rm[kNT];
  __shared__ long long s_rk[kNT];
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool large = false;
  int64_t turn = 0;
  for (int64_t t0 = (int64_t)blockIdx.x * kWarps; t0 < n_tiles; t0 += (int64_t)gridDim.x * kWarps, turn++) {
    const int64_t t = t0 + warp;
    const int ne = t < n_tiles ? events_of(A, t) : 0;
    int64_t lo = 0, hi = 0;
    if (lane < ne) {
      lo = A.off[t * A.tile + lane];
      hi = A.off[t * A.tile + lane + 1];
    }
    const bool bad = __any_sync(kAll, lane < ne && bad_event(A, t * A.tile + lane, lo, hi));
    if (!bad && ((rare >> (turn / A.turns)) & 1ull))
      warp_tile<LP, true>(A, T, reinterpret_cast<WarpBuf *>(s_dyn)[warp], s_hist, t * A.tile, ne, lo, hi);
    large |= !bad && lane < ne && hi - lo > kCap;
  }
  if (!__syncthreads_or(large)) return;
  ffm::EvPart *part = reinterpret_cast<ffm::EvPart *>(s_dyn);
  static_assert(sizeof(WarpBuf) * kWarps >= kNT * sizeof(ffm::EvPart), "an event staged by the block");
  int64_t counted = 0;
  for (int64_t t0 = (int64_t)blockIdx.x * kWarps; t0 < n_tiles; t0 += (int64_t)gridDim.x * kWarps) {
    const int64_t t = t0 + warp;
    const int ne = t < n_tiles ? events_of(A, t) : 0;
    bool bad = false;
    if (lane < ne) {
      const int64_t lo = A.off[t * A.tile + lane], hi = A.off[t * A.tile + lane + 1];
      bad = bad_event(A, t * A.tile + lane, lo, hi);
      s_off[warp][lane] = lo;
      if (lane == ne - 1) s_off[warp][ne] = hi;
    }
    bad = __any_sync(kAll, bad);
    if (lane == 0) s_ne[warp] = bad ? 0 : ne;
    __syncthreads();
    for (int w = 0; w < kWarps; w++) {
      for (int e = 0; e < s_ne[w]; e++) {
        const int64_t pb = s_off[w][e], n = s_off[w][e + 1] - pb, ev = (t0 + w) * A.tile + e;
        if (n <= kCap) continue;
        if (n <= kNT)
          staged_event_select<LP>(A, T, part, s_hist, pb, (int)n, &s_rd[threadIdx.x], &s_rk[threadIdx.x],
                                  &s_rm[threadIdx.x]);
        else
          big_event_select<LP>(A, T, s_hist, pb, n, &s_rd[threadIdx.x], &s_rk[threadIdx.x], &s_rm[threadIdx.x]);
        __syncthreads();
        if (threadIdx.x == 0) {
          double bd = s_rd[0], bm = s_rm[0];
          long long bk = s_rk[0];
          for (int u = 1; u < kNT; u++)
            if (better(s_rd[u], s_rk[u], bd, bk)) {
              bd = s_rd[u];
              bk = s_rk[u];
              bm = s_rm[u];
            }
          if (A.best_k) A.best_k[ev] = bk;
          if (A.best_m) A.best_m[ev] = bk >= 0 ? bm : NAN;
        }
        __syncthreads();
        counted = n > kNT ? 0 : counted + n * (n - 1) / 2;  // big_event_select has flushed
        if (counted >= kFlushPairs) {
          flush_slots(A, s_hist);
          __syncthreads();
          counted = 0;
        }
      }
    }
    __syncthreads();  // before the next tiles' offsets
  }
}

template <int LP>
__global__ void __launch_bounds__(kNT, 3) pair_select_kernel(const __grid_constant__ SArgs A) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  WarpBuf *bufs = reinterpret_cast<WarpBuf *>(s_dyn);
  unsigned *s_hist = reinterpret_cast<unsigned *>(bufs + kWarps);
  for (int s = threadIdx.x; s < A.n_bins + 2; s += kNT) s_hist[s] = 0u;
  __syncthreads();
  const ffm::LcTab T{ffm::kHypTab, ffm::kSinTab};  // read through L1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = (A.n_events + A.tile - 1) / A.tile;
  // a tile's offsets are loaded one tile ahead, and its particles' lines asked for then
  const auto offsets_of = [&](int64_t t, int64_t &lo, int64_t &hi) {
    lo = hi = 0;
    if (t < n_tiles && lane < events_of(A, t)) {
      lo = A.off[t * A.tile + lane];
      hi = A.off[t * A.tile + lane + 1];
    }
  };
  const int64_t step = (int64_t)gridDim.x * kWarps;
  int64_t t = (int64_t)blockIdx.x * kWarps + warp, lo, hi;
  bool large = false;
  unsigned long long rare = 0;  // the warp's tiles to walk again, one bit for 1/64 of them
  offsets_of(t, lo, hi);
  for (int64_t turn = 0; t < n_tiles; t += step, turn++) {
    int64_t lo1, hi1;
    offsets_of(t + step, lo1, hi1);
    if (t + step < n_tiles)
      prefetch_particles<LP>(A, __shfl_sync(kAll, lo1, 0), __shfl_sync(kAll, hi1, events_of(A, t + step) - 1));
    const int left = warp_tile<LP, false>(A, T, bufs[warp], s_hist, t * A.tile, events_of(A, t), lo, hi);
    large |= (left & kLarge) != 0;
    if (left & kRare) rare |= 1ull << (turn / A.turns);
    lo = lo1;
    hi = hi1;
  }
  if (__syncthreads_or(large || rare != 0)) finish_tiles<LP>(A, s_dyn, s_hist, n_tiles, rare);
  __syncthreads();
  flush_slots(A, s_hist);
}

template <int LP>
cudaError_t launch_l(SArgs A, cudaStream_t s) {
  constexpr auto k = pair_select_kernel<LP>;
  const size_t smem = kWarps * sizeof(WarpBuf) + (size_t)(A.n_bins + 2) * sizeof(unsigned);
  cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  // resident CTAs; a small call takes smaller tiles, so that its events reach all of their warps
  int per_sm = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kNT, smem);
  if (err != cudaSuccess) return err;
  const int64_t warps = (int64_t)num_sms() * (per_sm < 1 ? 1 : per_sm) * kWarps;
  const int64_t want = (A.n_events + warps - 1) / warps;
  A.tile = (int)(want < kMaxTile ? want : kMaxTile);
  const int64_t n_tiles = (A.n_events + A.tile - 1) / A.tile;
  const int64_t need = (n_tiles + kWarps - 1) / kWarps, cap = warps / kWarps;
  // the CTAs that fit at once; more where a warp would have more than kMaxTurns tiles (30 M events)
  const int64_t few = (n_tiles + kWarps * kMaxTurns - 1) / (kWarps * kMaxTurns);
  const int64_t grid = need < cap ? need : few > cap ? few : cap;
  A.turns = (int)((n_tiles + 64 * grid * kWarps - 1) / (64 * grid * kWarps));
  k<<<(unsigned)grid, kNT, smem, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_pair_select(const Lv &p, const int64_t *off, int64_t n_events,
                               int64_t n_particles, double pt_min, double eta_max, double lo,
                               double hi, int n_bins, double target, uint64_t *counts,
                               int64_t *best_k, double *best_m, cudaStream_t s) {
  SArgs A;
  A.p = p;
  A.off = off;
  A.n_events = n_events;
  A.n_particles = n_particles;
  A.cuts = make_cuts(pt_min, eta_max);
  A.lo = lo;
  A.hi = hi;
  A.inv_w = (double)n_bins / (hi - lo);
  A.target = target;
  A.n_bins = n_bins;
  // the float slot: lo in two floats, 1/width, and the absolute part of its error; a range or width
  // outside the floats leaves every pair to the FP64 slot (an infinite tolerance)
  const double inv_abs = fabs(A.inv_w), reach = fabs(lo) + fabs(hi);
  const bool fits = inv_abs > 1e-30 && inv_abs < 1e30 && reach < 1e30;
  A.lo_h = fits ? (float)lo : 0.0f;
  A.lo_l = fits ? (float)(lo - (double)A.lo_h) : 0.0f;
  A.inv_f = fits ? (float)A.inv_w : 0.0f;
  A.tol0 = fits ? (float)(reach * A.inv_w * 0x1p-40) + 0x1p-40f : INFINITY;
  A.counts = reinterpret_cast<unsigned long long *>(counts);
  A.best_k = best_k;
  A.best_m = best_m;
  A.status = device_status_word();
  return p.layout == GVX_SOA ? launch_l<GVX_SOA>(A, s) : launch_l<GVX_AOS>(A, s);
}

}  // namespace gvx
