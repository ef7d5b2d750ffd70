// slab.cuh -- device view of a slab problem and the per-particle physics
// shared by the history-based and the event-based slab schedules.
//
// Both schedules call the same functions below for every draw, flight,
// collision and tally contribution, so they make the same int64 tally
// contributions; int64 addition is associative, so the totals are
// bit-identical whatever the order of the additions.
//
// fp64 path: every operation is the one the transport definition names,
// rounded once (this file is compiled with --fmad=false, so no a*b+c is
// contracted).  fp32 path: flight length and geometry in fp32, with an fp64
// recomputation of the leak/collide decision when the fp32 end point lands
// within a guard band of a slab face; uniforms, absorption tests and the
// fixed-point scaling of tally contributions stay exact (fp64 or integer).
#pragma once
#include <cstdint>

#include "../../include/mc.h"
#include "mc_device.cuh"
#include "fp_exact.cuh"
#include "mc_log.cuh"

namespace mcs {

struct SlabDev {
  double L, sigma_t, c;
  uint64_t n_hist, seed, stride_q, id_offset, key, tally_offset;
  uint32_t n_bins, n_batches, source, seeding;
  // derived on the device by the prep kernel
  double h;             // bin width L / n_bins
  double inv_h;         // n_bins / L: candidate-bin lookup only
  uint32_t ih_q;        // inv_h as ih_q 2^-ih_s (the lookup on the integer pipes)
  int ih_s;
  double inv_st;        // 1 / sigma_t
  double p_abs;         // 1 - c
  uint64_t p_abs_n;     // ceil((1 - c) 2^53): u < 1 - c  <=>  n < p_abs_n for u = n 2^-53
  float guard_f;        // fp32 path: half-width of the fp64 guard band at a face
  float L_f, h_f, inv_h_f, inv_st_f;
  uint64_t seed_hash;   // hash seeding: seed half of hash(., s) or of hash(., hash(key, s))
  uint64_t hist_begin;  // global index of local history 0
  uint64_t tab_off;     // its edge table (n_bins + 1) and width table (n_bins) in the table
                        // area after the records, in doubles (set on the host)
};

constexpr double kFix = 4294967296.0;  // 2^32: fixed-point scale of the tallies

// One LCG stream (Eq. 1) and its draw counter, held in registers.
template <int M>
struct Rng {
  uint64_t x;
  uint64_t draws;
  __device__ __forceinline__ double next(const mcd::Lcg& l) {
    x = mcd::lcg_step(x, l.g, l.c);
    ++draws;
    return mcd::u01<M>(x, l.m);
  }
  // The same draw as its integer n (u = n 2^-53), for comparisons and exact
  // integer arithmetic on u.
  __device__ __forceinline__ uint64_t next_n(const mcd::Lcg& l) {
    x = mcd::lcg_step(x, l.g, l.c);
    ++draws;
    return mcd::u53<M>(x, l.m);
  }
};

// The state k steps after x through a table of the maps of 2^j steps.
__device__ __forceinline__ uint64_t skip_tab(const mcd::Affine* tab, uint64_t x, uint64_t k) {
  while (k) {
    const int j = __ffsll((long long)k) - 1;
    x = mcd::apply(tab[j], x);
    k &= k - 1;
  }
  return x;
}

// Seed of local history `id` (Eqs. 2-4): hash(id, s), hash(id, hash(key, s))
// or X_{Q * (id_offset + id)}.
__device__ __forceinline__ uint64_t slab_seed(const SlabDev& p, uint64_t id, const mcd::Affine* tab,
                                              uint64_t mask) {
  if (p.seeding == MC_SEED_STRIDE) return skip_tab(tab, p.seed, p.stride_q * (p.id_offset + id)) & mask;
  return mcd::hash_with(id, p.seed_hash) & mask;
}

// The processing order of a launch of several problems: problem order[k]'s
// histories take ticket positions [begin[k], begin[k + 1]) (the prep kernel
// ranks the problems by their expected flights per history, longest first,
// so that the long chains start early and do not form the launch's tail).
// An empty order (order == nullptr) takes the histories in id order from
// range_begin.  Either way history gi keeps its own stream, so the order
// changes no result.
struct Order {
  const uint32_t* order;
  const uint64_t* begin;
};

__device__ __forceinline__ uint32_t find_problem_of(const SlabDev* p, uint32_t n, uint64_t gi) {
  uint32_t lo = 0, hi = n - 1;  // largest i with hist_begin <= gi
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (p[mid].hist_begin <= gi) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Problem and global history index of ticket position t.
__device__ __forceinline__ void ticket_history(const SlabDev* p, uint32_t n, uint64_t range_begin, const Order& o,
                                               uint64_t t, uint32_t& pi, uint64_t& gi) {
  if (o.order) {
    uint32_t lo = 0, hi = n - 1;  // largest k with begin[k] <= t
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (o.begin[mid] <= t) lo = mid; else hi = mid - 1;
    }
    pi = o.order[lo];
    gi = p[pi].hist_begin + (t - o.begin[lo]);
    return;
  }
  gi = range_begin + t;
  pi = n == 1 ? 0u : find_problem_of(p, n, gi);
}

__device__ __forceinline__ uint64_t batch_of(uint64_t id, uint64_t n_hist, uint32_t n_batches) {
  // floor(id * n_batches / n_hist) without 128-bit arithmetic when it fits.
  if (id <= (~0ull) / (n_batches ? n_batches : 1)) return (id * n_batches) / n_hist;
  const unsigned __int128 t = (unsigned __int128)id * n_batches;
  return (uint64_t)(t / n_hist);
}

__device__ __forceinline__ double slab_edge(const SlabDev& p, int j) {
  if (j >= (int)p.n_bins) return p.L;
  return j < 2048 ? mcx::mul_small((uint32_t)j, p.h) : (double)j * p.h;  // RN(j h)
}

// A bin index within one of floor(x n_bins / L), x >= 0 (integer pipes).
__device__ __forceinline__ int bin_guess(const SlabDev& p, double x) {
  return (int)min(mcx::guess_floor_mul(x, p.ih_q, p.ih_s), (uint64_t)p.n_bins);
}

__device__ __forceinline__ int clamp_bin(int j, int nb) { return j < 0 ? 0 : (j >= nb ? nb - 1 : j); }

// Tally sink: this history's [bin] row in shared memory (the whole tally
// staged) or global memory, the offset of its warp's row cache in dynamic
// shared memory (kNoRow: none) where the warp accumulates that row, and an
// optional table of the bin edges e_0..e_nb (nullptr: each edge is computed
// as j * h).
constexpr uint32_t kNoRow = ~0u;
struct Sink {
  unsigned long long* base;
  const double* edges;
  const double* widths;  // with edges: widths[j] = e_{j+1} - e_j (the same fp64 difference)
  bool agg;              // warp-aggregated atomics (mcd::warp_agg_add) instead of one per lane
  uint32_t row = kNoRow;
  __device__ __forceinline__ void add(int j, long long v) const {
    if (row != kNoRow) {
      extern __shared__ unsigned long long s_dyn[];
      atomicAdd(s_dyn + row + j, (unsigned long long)v);
    } else if (agg) {
      mcd::warp_agg_add(base + j, (unsigned long long)v);
    } else {
      atomicAdd(base + j, (unsigned long long)v);
    }
  }
};

// Order of two non-negative doubles from their bit patterns (IEEE-754
// orders non-negative values like their bits read as integers): the fp64
// comparisons of the path run on the integer pipes.
__device__ __forceinline__ bool nn_lt(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}

__device__ __forceinline__ double edge_of(const SlabDev& p, const Sink& s, int j) {
  return s.edges ? s.edges[j] : slab_edge(p, j);
}

// The bin of a position x in [0, L]: the largest j with e_j <= x (the last
// bin for x = L).
__device__ __forceinline__ int bin_of(const SlabDev& p, const Sink& s, double x) {
  const int nb = (int)p.n_bins;
  int j = clamp_bin(bin_guess(p, x), nb);
  while (j > 0 && nn_lt(x, edge_of(p, s, j))) --j;
  while (j + 1 < nb && !nn_lt(x, edge_of(p, s, j + 1))) ++j;
  return j;
}

// Track length in every bin met by a flight from x to xe (both in [0, L];
// forward: xe >= x, else xe <= x): |[x, xe] & [e_j, e_{j+1}]| / |mu|, to fixed
// point.  w_fix = 2^32 / |mu|, rounded once; since scaling by 2^32 commutes
// with rounding, (hi - lo) * w_fix rounds to exactly 2^32 times the rounded
// (hi - lo) * (1/|mu|).  The walk starts from x's bin j, goes the way the
// particle flies and leaves j at the bin of xe, where the next flight starts:
// no bin is ever looked up.  (At an edge either neighbour will do for j: the
// piece in the other one has length zero and adds nothing.)  It goes piece by
// piece, so that a caller can stop between two: walk_first adds the piece to
// xe or to the first edge, walk_next the next one, to xe or a whole bin with
// its length from the width table; both return whether pieces are left.
// ADD: a piece is rounded by an addition instead of from its bits, one fp64
// instruction for some 15 integer ones.  The history kernel is bound by issue
// (slab_long 141 -> 137 ms, 300 000 histories of 9 flights 253 -> 243 us); the
// event schedule waits for its bank and its latency grows (97.8 -> 100.3 ms).
template <bool ADD>
struct Walk64 {
  double xe, w;  // the end, and 2^32 / |mu|
  bool fwd;
};
template <bool ADD>
__device__ __forceinline__ long long walk_fix(double v) {
  return ADD ? mcx::llrint_add(v) : mcx::llrint_nonneg(v);
}
template <bool ADD>
__device__ __forceinline__ bool walk_first(const SlabDev& p, double x, const Walk64<ADD>& k, const Sink& s, int j) {
  const double e = edge_of(p, s, j + (k.fwd ? 1 : 0));
  const bool last = k.fwd ? !nn_lt(e, k.xe) : !nn_lt(k.xe, e);
  s.add(j, walk_fix<ADD>(__dmul_rn(mcx::abs_bits(__dsub_rn(last ? k.xe : e, x)), k.w)));
  return !last;
}
template <bool ADD>
__device__ __forceinline__ bool walk_next(const SlabDev& p, const Walk64<ADD>& k, const Sink& s, int& j) {
  j += k.fwd ? 1 : -1;
  const double e0 = edge_of(p, s, j + (k.fwd ? 0 : 1)), e1 = edge_of(p, s, j + (k.fwd ? 1 : 0));
  const bool last = k.fwd ? !nn_lt(e1, k.xe) : !nn_lt(k.xe, e1);
  const double len = !last && s.widths ? s.widths[j] : mcx::abs_bits(__dsub_rn(last ? k.xe : e1, e0));
  s.add(j, walk_fix<ADD>(__dmul_rn(len, k.w)));
  return !last;
}

// Exact llrint((double)v * 2^32) for a finite float v >= 0 (scaling by 2^32
// is exact; bits below the last are rounded half to even).
// On integers, for any v.  Out of line: tracks below 2^22 cm take the other way.
static __device__ __noinline__ long long fix32_any(float v) {
  const uint32_t b = __float_as_uint(v);
  const int e = (int)(b >> 23) & 0xff;
  if (e == 0) return 0;  // zero or subnormal: below 2^-126, rounds to 0 at scale 2^32
  const uint64_t mant = (uint64_t)((b & 0x7fffffu) | 0x800000u);
  const int sh = e - 127 - 23 + 32;  // value * 2^32 = mant * 2^sh
  if (sh >= 0) return (long long)(mant << sh);
  if (sh < -25) return 0;
  const int r = -sh;
  const uint64_t q = mant >> r, rem = mant & ((1ull << r) - 1ull), half = 1ull << (r - 1);
  const uint64_t up = (rem > half) || (rem == half && (q & 1ull));
  return (long long)(q + up);
}

// For v < 2^22 on the fp32 pipe, without branches: adding 2^23 rounded down
// leaves floor(v) in the low bits; the fraction (exact) gives its next 16
// bits the same way, and the last 16 by an addition rounded to nearest even,
// whose parity is that of the whole.  The last 16 can round up to 2^16 (v =
// 2^-16 - 2^-40): the low word is a sum, which carries that into the bits
// above.  It cannot carry out of the low word: that takes a fraction of 33
// leading ones, and a fraction has at most 24 bits.
__device__ __forceinline__ long long fix32_from_float(float v) {
  if (v >= 4194304.0f) return fix32_any(v);
  constexpr float kM = 8388608.0f;  // 2^23, bit pattern 0x4b000000
  const float m1 = __fadd_rz(v, kM);
  const float g = __fmul_rn(__fsub_rn(v, __fsub_rn(m1, kM)), 65536.0f);
  const float m2 = __fadd_rz(g, kM);
  const float m3 = __fadd_rn(__fmul_rn(__fsub_rn(g, __fsub_rn(m2, kM)), 65536.0f), kM);
  const uint32_t lo = __float_as_uint(m2) * 65536u + (__float_as_uint(m3) - 0x4b000000u);
  return (long long)(((uint64_t)(__float_as_uint(m1) - 0x4b000000u) << 32) | lo);
}

__device__ __forceinline__ float slab_edge_f(const SlabDev& p, int j) {
  return j >= (int)p.n_bins ? p.L_f : (float)j * p.h_f;
}

// The fp32 path's positions are pairs of floats.  Each bin's length is taken
// from the pairs, (hi_h - lo_h) + (hi_l - lo_l), so a flight whose
// displacement is far below an ulp of its position (a direction nearly
// parallel to the faces, where 1 / |mu| is large) keeps its true length
// instead of an ulp of the position times 1 / |mu|.
__device__ __forceinline__ int bin_of_pair(const SlabDev& p, float h, float l) {
  // the largest j with e_j <= h + l (fp32 edges), from the scaled guess
  const int nb = (int)p.n_bins;
  int j = clamp_bin((int)(h * p.inv_h_f), nb);
  while (j > 0) {
    const float e = slab_edge_f(p, j);
    if (h < e || (h == e && l < 0.0f)) --j; else break;
  }
  while (j + 1 < nb) {
    const float e = slab_edge_f(p, j + 1);
    if (h > e || (h == e && l >= 0.0f)) ++j; else break;
  }
  return j;
}

// The fp32 walk, to the pair (eh + el) with weight w = 1 / |mu|.
struct Walk32 {
  float eh, el, w;
  bool fwd;
};
__device__ __forceinline__ bool walk_piece(const SlabDev& p, float xh, float xl, const Walk32& k, const Sink& s, int j) {
  const float e = slab_edge_f(p, j + (k.fwd ? 1 : 0));
  // the end lies beyond the edge?
  const bool last = k.fwd ? !(k.eh > e || (k.eh == e && k.el > 0.0f)) : !(k.eh < e || (k.eh == e && k.el < 0.0f));
  const float th = last ? k.eh : e, tl = last ? k.el : 0.0f;
  const float d = __fadd_rn(__fsub_rn(th, xh), __fsub_rn(tl, xl)), len = k.fwd ? d : -d;
  if (len > 0.0f) s.add(j, fix32_from_float(__fmul_rn(len, k.w)));
  return !last;
}
__device__ __forceinline__ bool walk_first(const SlabDev& p, float xh, float xl, const Walk32& k, const Sink& s,
                                           int j) {
  return walk_piece(p, xh, xl, k, s, j);
}
__device__ __forceinline__ bool walk_next(const SlabDev& p, const Walk32& k, const Sink& s, int& j) {
  j += k.fwd ? 1 : -1;
  return walk_piece(p, slab_edge_f(p, j + (k.fwd ? 0 : 1)), 0.0f, k, s, j);
}

__device__ __forceinline__ void point32(const SlabDev& p, float x, float d, const Sink& s) {
  const int nb = (int)p.n_bins;
  int j = clamp_bin((int)(x * p.inv_h_f), nb);
  while (j > 0 && x < slab_edge_f(p, j)) --j;
  while (j + 1 < nb && x >= slab_edge_f(p, j + 1)) ++j;
  s.add(j, fix32_from_float(d));
}

// Particle state of the slab physics.  fp64 path: x, mu and w_mu, which
// holds 2^32 / |mu| (0 for mu = 0); the fp32 path keeps its geometry in
// fp32: the position as an unevaluated sum xf + xlo of two floats (so that
// it does not drift from the fp64 trajectory by one rounding per flight),
// muf and wf = 1 / |muf|.  Both keep the bin of the position.
struct SlabParticle {
  double x, mu, w_mu;
  float xf, xlo, muf, wf;
  int j;  // the bin of the position
};

// s + t = a + b exactly (Knuth's TwoSum; six fp32 operations, no fused
// multiply-add, so every one rounds once).
__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& t) {
  s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bv)), __fsub_rn(b, bv));
}

// z 2^-64 rounded once to fp32, for z != 0 with its low 10 bits zero: the
// leading 32 bits of z, with a sticky bit for the rest, through the 32-bit
// conversion.  The same value as rounding the exact double (which costs the
// fp64 unit 16 cycles per SM and warp); z below 2^32 takes that way.
__device__ __forceinline__ float top_bits_to_float(uint64_t z) {
  const uint32_t hi = (uint32_t)(z >> 32), lo = (uint32_t)z;
  if (hi == 0u) return __uint2float_rn(lo) * 0x1p-64f;  // at most 22 bits: exact
  const int lz = __clz((int)hi);
  const uint32_t t = __funnelshift_l(lo, hi, lz) | ((lo << lz) != 0u ? 1u : 0u);
  return __int_as_float(__float_as_int(__uint2float_rn(t)) - ((32 + lz) << 23));
}

// The uniform u = n 2^-53 (n < 2^53) rounded once to fp32.
__device__ __forceinline__ float u53_to_float(uint64_t n) { return top_bits_to_float(n << 11); }

// -ln(1 - u) in fp32 for u = n 2^-53: log1pf(-u) below 1/2 (no
// cancellation for small u), else logf of 1 - u, which is exact as an
// integer and at least 2^-53, so it rounds to a positive float and the result
// is finite (log1pf of -(float)u would meet -1 and give an infinite distance
// for u within 2^-25 of 1).
__device__ __forceinline__ float flight_f32(uint64_t n) {
  const bool low = n < (1ull << 52);
  const float v = u53_to_float(low ? n : (1ull << 53) - n);
  return low ? -log1pf(-v) : -logf(v);
}

// The fp32 direction 2u - 1 for u = n 2^-53, rounded once.
__device__ __forceinline__ float mu_f32(uint64_t n) {
  const long long w = (long long)(n << 1) - (1ll << 53);
  if (w == 0) return 0.0f;
  const float a = 2.0f * top_bits_to_float((uint64_t)(w < 0 ? -w : w) << 10);
  return w < 0 ? -a : a;
}

// 2^32 / |mu| rounded once: 2^32 RN(1 / |mu|), the reciprocal on the
// integer pipes (fp_exact.cuh), the scaling an exponent add.
__device__ __forceinline__ double fix_per_mu(double mu) {
  const double w = mcx::scale_pow2(mcx::recip_normal(mcx::abs_bits(mu)), 32);
  return mcx::d_zero(mu) ? 0.0 : w;
}

// Per-lane counters for the lane's current problem (flushed with atomics,
// lane by lane or summed over a converged warp first: a problem's counters
// share a cache line).
struct LaneCounts {
  int prob;
  uint32_t src, flights, coll, absn, scat, llo, lhi, capped, exh;
  uint64_t draws, exd, maxd;
  __device__ void clear() {
    src = flights = coll = absn = scat = llo = lhi = capped = exh = 0u;
    draws = exd = maxd = 0ull;
  }
  __device__ void flush(unsigned long long* counts) {
    if (prob < 0) return;
    unsigned long long* c = counts + (size_t)prob * MC_NCOUNT;
    if (src) atomicAdd(c + MC_C_SOURCE, (unsigned long long)src);
    if (flights) atomicAdd(c + MC_C_FLIGHTS, (unsigned long long)flights);
    if (coll) atomicAdd(c + MC_C_COLLISIONS, (unsigned long long)coll);
    if (absn) atomicAdd(c + MC_C_ABSORPTIONS, (unsigned long long)absn);
    if (scat) atomicAdd(c + MC_C_SCATTERS, (unsigned long long)scat);
    if (llo) atomicAdd(c + MC_C_LEAK_LO, (unsigned long long)llo);
    if (lhi) atomicAdd(c + MC_C_LEAK_HI, (unsigned long long)lhi);
    if (draws) atomicAdd(c + MC_C_DRAWS, (unsigned long long)draws);
    if (exh) atomicAdd(c + MC_C_EXCEED_HIST, (unsigned long long)exh);
    if (exd) atomicAdd(c + MC_C_EXCEED_DRAWS, (unsigned long long)exd);
    if (capped) atomicAdd(c + MC_C_CAPPED, (unsigned long long)capped);
    if (maxd) atomicMax(c + MC_C_MAX_DRAWS, (unsigned long long)maxd);
    clear();
  }
  // The same for a whole converged warp: sums first, then one lane's atomics.
  __device__ void flush_warp(unsigned long long* counts) {
    const int p = mcd::warp_common_prob(prob);
    if (p == -2) { flush(counts); return; }
    if (p < 0) return;
    const unsigned long long so = mcd::warp_sum64(src), fl = mcd::warp_sum64(flights), co = mcd::warp_sum64(coll),
                             ab = mcd::warp_sum64(absn), sc = mcd::warp_sum64(scat), lo = mcd::warp_sum64(llo),
                             hi = mcd::warp_sum64(lhi), cp = mcd::warp_sum64(capped), ex = mcd::warp_sum64(exh),
                             dr = mcd::warp_sum64(draws), ed = mcd::warp_sum64(exd), mx = mcd::warp_max64(maxd);
    if ((threadIdx.x & 31u) == 0u) {
      unsigned long long* c = counts + (size_t)p * MC_NCOUNT;
      if (so) atomicAdd(c + MC_C_SOURCE, so);
      if (fl) atomicAdd(c + MC_C_FLIGHTS, fl);
      if (co) atomicAdd(c + MC_C_COLLISIONS, co);
      if (ab) atomicAdd(c + MC_C_ABSORPTIONS, ab);
      if (sc) atomicAdd(c + MC_C_SCATTERS, sc);
      if (lo) atomicAdd(c + MC_C_LEAK_LO, lo);
      if (hi) atomicAdd(c + MC_C_LEAK_HI, hi);
      if (dr) atomicAdd(c + MC_C_DRAWS, dr);
      if (ex) atomicAdd(c + MC_C_EXCEED_HIST, ex);
      if (ed) atomicAdd(c + MC_C_EXCEED_DRAWS, ed);
      if (cp) atomicAdd(c + MC_C_CAPPED, cp);
      if (mx) atomicMax(c + MC_C_MAX_DRAWS, mx);
    }
    clear();
  }
};

// Outcome of a flight or a collision.
enum Outcome : int { kContinue = 0, kAbsorbed = 1, kLeakLo = 2, kLeakHi = 3, kCollide = 4 };

// A new direction from its draw: mu and 2^32 / |mu|, or the fp32 pair.
template <bool F32>
__device__ __forceinline__ void set_direction(SlabParticle& q, uint64_t n) {
  if constexpr (!F32) {
    q.mu = mcx::two_u_minus_1(n);
    q.w_mu = fix_per_mu(q.mu);
  } else {
    q.muf = mu_f32(n);
    q.wf = q.muf != 0.0f ? __frcp_rn(fabsf(q.muf)) : 0.0f;
  }
}

// Source of a history (isotropic uniform in [0, L], or a beam at x = 0).
template <int M, bool F32>
__device__ __forceinline__ void slab_source(const SlabDev& p, Rng<M>& r, const mcd::Lcg& l, SlabParticle& q) {
  if (p.source == MC_SRC_BEAM) {
    q.x = 0.0; q.mu = 1.0; q.w_mu = kFix;
    q.xf = 0.0f; q.xlo = 0.0f; q.muf = 1.0f; q.wf = 1.0f;
    return;
  }
  const double u1 = r.next(l);
  if constexpr (!F32) {
    q.x = __dmul_rn(p.L, u1);
  } else {
    // x = L u as the fp64 path has it, split into two floats
    const double x64 = __dmul_rn(p.L, u1);
    q.xf = __double2float_rn(x64);
    q.xlo = __double2float_rn(__dsub_rn(x64, (double)q.xf));
  }
  set_direction<F32>(q, r.next_n(l));
}

// The end of a flight of the fp64 path: xn = x + pm (pm = d mu, rounded
// once), and whether it leaves the slab.  mu is never -0 (2u - 1 rounds an
// exact zero to +0), so its sign is the sign of its bit pattern; x, L and
// the positions of a forward flight are non-negative.
__device__ __forceinline__ int advance64(const SlabDev& p, double x, double mu, double pm, double& xn) {
  xn = __dadd_rn(x, pm);
  const long long mb = __double_as_longlong(mu);
  if (mb > 0 && !nn_lt(xn, p.L)) return kLeakHi;
  if (mb < 0 && __double_as_longlong(xn) <= 0) return kLeakLo;
  return kCollide;
}

// The tally of that flight, from x's bin j: the track from x to xn, to the
// face it leaves through, or (mu = 0) the whole distance d in the bin holding
// x.  Every kind of flight ends in the one walk, with its end chosen first, so
// that the lanes of a warp whose flights differ in kind still walk the bins
// together.  begin_tally adds the first piece and returns whether walk_next
// has more (which leaves j at the bin of xn); tally64 adds them all.
template <bool ADD>
__device__ __forceinline__ bool begin_tally(const SlabDev& p, double x, double xn, double mu, double d, double w_mu,
                                            int outcome, const Sink& s, int& j, Walk64<ADD>& k) {
  const long long mb = __double_as_longlong(mu);
  if (outcome == kCollide && mb == 0) {
    s.add(bin_of(p, s, x), mcx::fix32_nonneg(d));
    return false;
  }
  k.xe = outcome == kLeakHi ? p.L : (outcome == kLeakLo ? 0.0 : xn);
  k.w = w_mu;
  k.fwd = mb > 0;
  return walk_first(p, x, k, s, j);
}
__device__ __forceinline__ void tally64(const SlabDev& p, double x, double xn, double mu, double d, double w_mu,
                                        int outcome, const Sink& s, int& j) {
  Walk64<false> k;
  if (begin_tally(p, x, xn, mu, d, w_mu, outcome, s, j, k))
    while (walk_next(p, k, s, j)) {}
}

// The fp32 path's position step: xn + xnlo = (xf + xlo) + d muf, with pr =
// d muf rounded and pe its exact error (a fused multiply-add); the sum by
// TwoSum, the low parts' sum rounded once more (a second-order error).
__device__ __forceinline__ void pair_step(float xf, float xlo, float pr, float pe, float& xn, float& xnlo) {
  float s0, t0;
  two_sum_f(xf, pr, s0, t0);
  two_sum_f(s0, __fadd_rn(t0, __fadd_rn(xlo, pe)), xn, xnlo);
}

// The pair's end point is inside the slab and outside the guard bands: the
// flight collides there (advance32 decides the same, with the same xn, xnlo).
__device__ __forceinline__ bool plain_collision32(const SlabDev& p, float muf, float xn, float xnlo) {
  const bool near_hi = muf > 0.0f && fabsf(xn - p.L_f) <= p.guard_f;
  const bool near_lo = muf < 0.0f && fabsf(xn) <= p.guard_f;
  const bool leak_hi = muf > 0.0f && (xn > p.L_f || (xn == p.L_f && xnlo >= 0.0f));
  const bool leak_lo = muf < 0.0f && (xn < 0.0f || (xn == 0.0f && xnlo <= 0.0f));
  return !(near_hi | near_lo | leak_hi | leak_lo);
}

// The end of a flight of the fp32 path by pair_step, and whether it leaves
// the slab; near a face the leak-or-collide decision is made again in fp64
// from the flight's uniform nf() 2^-53 (called only there).
template <class UF>
__device__ __forceinline__ int advance32(const SlabDev& p, float xf, float xlo, float muf, float pr, float pe,
                                         UF nf, float& xn, float& xnlo) {
  pair_step(xf, xlo, pr, pe, xn, xnlo);
  // Guard band: re-decide leak vs collide in fp64 near a face.
  const bool near_hi = muf > 0.0f && fabsf(xn - p.L_f) <= p.guard_f;
  const bool near_lo = muf < 0.0f && fabsf(xn) <= p.guard_f;
  // xn + xnlo >= L (or <= 0) from the pair: the low part decides a tie of the high part
  bool leak_hi = muf > 0.0f && (xn > p.L_f || (xn == p.L_f && xnlo >= 0.0f));
  bool leak_lo = muf < 0.0f && (xn < 0.0f || (xn == 0.0f && xnlo <= 0.0f));
  if (near_hi || near_lo) {
    const double d64 = __dmul_rn(mclog::neglog1m_n(nf()), p.inv_st);
    const double x64 = __dadd_rn((double)xf, (double)xlo);
    const double xn64 = __dadd_rn(x64, __dmul_rn(d64, (double)muf));
    leak_hi = muf > 0.0f && xn64 >= p.L;
    leak_lo = muf < 0.0f && xn64 <= 0.0;
    xn = __double2float_rn(xn64);
    if (!leak_hi && !leak_lo) {
      // keep the collision site's high part strictly inside
      if (xn >= p.L_f) xn = __int_as_float(__float_as_int(p.L_f) - 1);
      if (xn <= 0.0f) xn = 1.0e-30f;
    }
    xnlo = __double2float_rn(__dsub_rn(xn64, (double)xn));
  }
  return leak_hi ? kLeakHi : (leak_lo ? kLeakLo : kCollide);
}

// Their counterparts for the fp32 path, on position pairs.  A pair's last
// rounding can move a flight of next to no length backwards; its bin is then
// looked up again.
__device__ __forceinline__ bool begin_tally(const SlabDev& p, float xf, float xlo, float xn, float xnlo, float muf,
                                            float d, float wf, int outcome, const Sink& s, int& j, Walk32& k) {
  if (outcome == kCollide && muf == 0.0f) {
    point32(p, xf, d, s);
    return false;
  }
  k.eh = xn;
  k.el = xnlo;
  if (outcome == kLeakHi) { k.eh = p.L_f; k.el = 0.0f; }
  else if (outcome == kLeakLo) { k.eh = 0.0f; k.el = 0.0f; }
  k.w = wf;
  k.fwd = muf > 0.0f;
  const bool more = walk_first(p, xf, xlo, k, s, j);
  const bool less = xn < xf || (xn == xf && xnlo < xlo), beyond = xn > xf || (xn == xf && xnlo > xlo);
  if (outcome == kCollide && (k.fwd ? less : beyond)) j = bin_of_pair(p, xn, xnlo);
  return more;
}
__device__ __forceinline__ void tally32(const SlabDev& p, float xf, float xlo, float xn, float xnlo, float muf,
                                        float d, float wf, int outcome, const Sink& s, int& j) {
  Walk32 k;
  if (begin_tally(p, xf, xlo, xn, xnlo, muf, d, wf, outcome, s, j, k))
    while (walk_next(p, k, s, j)) {}
}

template <bool F32> struct WalkOf { using type = Walk64<true>; };
template <> struct WalkOf<true> { using type = Walk32; };

// The bin of the particle's position, where none is known from a flight.
template <bool F32>
__device__ __forceinline__ int locate(const SlabDev& p, const SlabParticle& q, const Sink& s) {
  if constexpr (F32) return bin_of_pair(p, q.xf, q.xlo);
  else return bin_of(p, s, q.x);
}

// One flight from the particle's bin q.j: sample the distance, tally the
// track, and either leak (kLeakLo / kLeakHi) or stop at the collision site
// (kCollide).
template <int M, bool F32>
__device__ __forceinline__ int slab_flight(const SlabDev& p, Rng<M>& r, const mcd::Lcg& l, SlabParticle& q,
                                           const Sink& s) {
  if constexpr (!F32) {
    const double d = __dmul_rn(mclog::neglog1m_n(r.next_n(l)), p.inv_st);
    double xn;
    const int f = advance64(p, q.x, q.mu, __dmul_rn(d, q.mu), xn);
    tally64(p, q.x, xn, q.mu, d, q.w_mu, f, s, q.j);
    if (f == kCollide) q.x = xn;
    return f;
  } else {
    const uint64_t n = r.next_n(l);
    const float d = flight_f32(n) * p.inv_st_f;
    const float pr = __fmul_rn(d, q.muf);
    const float pe = __fmaf_rn(d, q.muf, -pr);
    float xn, xnlo;
    const int f = advance32(p, q.xf, q.xlo, q.muf, pr, pe, [n] { return n; }, xn, xnlo);
    tally32(p, q.xf, q.xlo, xn, xnlo, q.muf, d, q.wf, f, s, q.j);
    if (f == kCollide) {
      q.xf = xn;
      q.xlo = xnlo;
    }
    return f;
  }
}

// One collision at the current site: absorption (kAbsorbed) or isotropic
// scattering into a new direction (kContinue).
template <int M, bool F32>
__device__ __forceinline__ int slab_collide(const SlabDev& p, Rng<M>& r, const mcd::Lcg& l, SlabParticle& q) {
  if (r.next_n(l) < p.p_abs_n) return kAbsorbed;  // u < 1 - c
  set_direction<F32>(q, r.next_n(l));
  return kContinue;
}

// One event of the history schedule on the stream state x: a flight and, if
// the particle stays in the slab, a collision.  The event's three draws have
// fixed roles (distance, absorption test, new direction), so the new
// direction and its tally weight are computed beside the distance whether or
// not the event comes to use them: the two chains of integer operations
// (the logarithm, the reciprocal) are independent and fill each other's
// latencies.  x moves on by the draws the event takes.
// The tally gets its first piece; `more` says whether k has others, without
// which q.j is not yet the particle's bin.
template <int M, bool F32>
__device__ __forceinline__ int slab_event(const SlabDev& p, uint64_t& x, const mcd::Lcg& l, SlabParticle& q,
                                          const Sink& s, typename WalkOf<F32>::type& k, bool& more) {
  const uint64_t x1 = mcd::lcg_step(x, l.g, l.c), x2 = mcd::lcg_step(x1, l.g, l.c), x3 = mcd::lcg_step(x2, l.g, l.c);
  const uint64_t n = mcd::u53<M>(x1, l.m);
  SlabParticle nq = q;
  set_direction<F32>(nq, mcd::u53<M>(x3, l.m));
  int f;
  if constexpr (!F32) {
    asm volatile("" : "+d"(nq.mu), "+d"(nq.w_mu));  // not moved to its use after the tally
    const double d = __dmul_rn(mclog::neglog1m_n(n), p.inv_st);
    f = advance64(p, q.x, q.mu, __dmul_rn(d, q.mu), nq.x);
    more = begin_tally(p, q.x, nq.x, q.mu, d, q.w_mu, f, s, nq.j, k);
  } else {
    asm volatile("" : "+f"(nq.muf), "+f"(nq.wf));
    const float d = flight_f32(n) * p.inv_st_f;
    const float pr = __fmul_rn(d, q.muf);
    const float pe = __fmaf_rn(d, q.muf, -pr);
    f = advance32(p, q.xf, q.xlo, q.muf, pr, pe, [n] { return n; }, nq.xf, nq.xlo);
    more = begin_tally(p, q.xf, q.xlo, nq.xf, nq.xlo, q.muf, d, q.wf, f, s, nq.j, k);
  }
  q.j = nq.j;
  if (f != kCollide) {
    x = x1;
    return f;
  }
  if (mcd::u53<M>(x2, l.m) < p.p_abs_n) {  // u < 1 - c
    x = x2;
    return kAbsorbed;
  }
  x = x3;
  q = nq;
  return kContinue;
}

// Draws of a history of the slab: the source's (none for a beam), three per
// event, less those its last event did not take (event cap: whole events).
__device__ __forceinline__ uint64_t slab_draws(const SlabDev& p, uint64_t events, int outcome) {
  const uint64_t unused = outcome == kLeakLo || outcome == kLeakHi ? 2u : (outcome == kAbsorbed ? 1u : 0u);
  return (p.source == MC_SRC_BEAM ? 0u : 2u) + 3ull * events - unused;
}

}  // namespace mcs
