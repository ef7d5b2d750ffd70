// slab.cu -- persistent history-based slab transport and the host side of
// mc_transport_run.
//
// One lane carries one history at a time: its LCG state, position and
// direction stay in registers.  Each loop iteration every live lane flies
// one flight (and collides once); a lane whose history ended refills from
// its warp's chunk of history indices, and the warp leader takes a new chunk
// from a global ticket when the chunk runs dry.  So a warp keeps its lanes
// busy until the ticket is exhausted, however uneven the histories; the long
// ones that are left then are finished by the whole block together.
//
// Tallies are int64 fixed point (2^32), staged in shared memory when the
// whole tally fits and flushed with one global atomic per nonzero slot per
// block; otherwise each warp caches the tally row most of its lanes are on,
// and other contributions go to global atomics.  Counters are accumulated
// per lane and flushed when a lane changes problem.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "internal.h"
#include "slab.cuh"
#include "transport.h"

namespace {

using mcs::SlabDev;

// Bin edge and width tables of one problem, by the threads of a block.
__device__ __forceinline__ void write_tables(const SlabDev& q, double* __restrict__ tables) {
  double* e = tables + q.tab_off;
  double* w = e + q.n_bins + 1;
  for (uint32_t j = threadIdx.x; j <= q.n_bins; j += blockDim.x) e[j] = mcs::slab_edge(q, (int)j);
  for (uint32_t j = threadIdx.x; j < q.n_bins; j += blockDim.x)
    w[j] = __dsub_rn(mcs::slab_edge(q, (int)j + 1), mcs::slab_edge(q, (int)j));
}

// Bin edge and width tables of every problem, after the records (`tables`
// may be null: no tables).
__global__ void slab_tables_kernel(const SlabDev* __restrict__ p, uint32_t n, double* __restrict__ tables) {
  for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) write_tables(p[i], tables);
}

// Expected flights per history of a slab problem with a uniform isotropic
// source, a ranking key only: the first-flight escape probability of such a
// source in a slab of optical thickness tau is (1 - 2 E3(tau)) / (2 tau)
// (E3 approximated by exp(-tau) / (tau + 2)), every later flight is taken to
// escape as often, and a collision continues with probability c:
// 1 / (1 - c (1 - P_esc)).
__device__ __forceinline__ float expected_flights(const SlabDev& q) {
  const float tau = fmaxf((float)(q.L * q.sigma_t), 1e-6f);
  const float e3 = __expf(-tau) / (tau + 2.0f);
  const float p_esc = fminf(1.0f, (1.0f - 2.0f * e3) / (2.0f * tau));
  return 1.0f / fmaxf(1e-6f, 1.0f - (float)q.c * (1.0f - p_esc));
}

// The fields of a record that follow from the others (but hist_begin).
__device__ __forceinline__ void derive(SlabDev& q) {
  q.h = q.L / (double)q.n_bins;
  q.inv_h = (double)q.n_bins / q.L;
  mcx::fixed_of(q.inv_h, q.ih_q, q.ih_s);
  q.inv_st = 1.0 / q.sigma_t;
  q.p_abs = 1.0 - q.c;
  q.p_abs_n = (uint64_t)ceil(q.p_abs * 0x1p53);
  q.L_f = (float)q.L;
  q.h_f = q.L_f / (float)q.n_bins;
  q.inv_h_f = (float)q.n_bins / q.L_f;
  q.inv_st_f = 1.0f / (float)q.sigma_t;
  q.guard_f = q.L_f * 0x1p-18f;
  const uint64_t parent = q.seeding == MC_SEED_HASH_HIER ? mcd::hash64(q.key, q.seed) : q.seed;
  q.seed_hash = mcd::seed_hash_of(parent);
}

// hist_begin of every record and (order non-null) the processing order, by
// one block, from records whose other fields are complete.
__device__ __forceinline__ void chain_records(SlabDev* __restrict__ p, uint32_t n, uint32_t* __restrict__ order,
                                              uint64_t* __restrict__ order_begin) {
  if (threadIdx.x == 0) {
    uint64_t acc = 0;
    for (uint32_t i = 0; i < n; ++i) {
      p[i].hist_begin = acc;
      acc += p[i].n_hist;
    }
  }
  if (!order) return;
  // rank by expected flights, descending; ties by index (a stable order)
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
    const float fi = expected_flights(p[i]);
    uint32_t r = 0;
    for (uint32_t j = 0; j < n; ++j) {
      const float fj = expected_flights(p[j]);
      r += (fj > fi || (fj == fi && j < i)) ? 1u : 0u;
    }
    order[r] = i;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t acc = 0;
    for (uint32_t k = 0; k < n; ++k) {
      order_begin[k] = acc;
      acc += p[order[k]].n_hist;
    }
    order_begin[n] = acc;
  }
}

__global__ void slab_prep_kernel(SlabDev* __restrict__ p, uint32_t n, uint32_t* __restrict__ order,
                                 uint64_t* __restrict__ order_begin) {
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) derive(p[i]);
  __syncthreads();
  chain_records(p, n, order, order_begin);
}

// A whole call's set-up in one launch, for few problems (their records travel
// with the launch's arguments): records, order and tables as slab_prep has
// them, the ticket, and a fresh tally's zeros.  Against an upload from pinned
// memory, two prep kernels and three memsets, a call of 10^4 histories whose
// problem differs from the last one's took 59 us and takes 38 (6 of them by
// slab_history_kernel_few).
struct InitArgs {
  SlabDev src[mci::kInitProblems];
  uint32_t n;
  SlabDev* dst;
  uint32_t* order;          // nullable
  uint64_t* order_begin;
  double* tables;           // nullable
  unsigned long long* ticket;
  unsigned long long* bins;    // nullable: accumulating
  unsigned long long* counts;
  uint64_t n_slots;
};

__global__ void __launch_bounds__(128) slab_init_kernel(const InitArgs a) {
  const uint32_t tblocks = a.tables ? a.n : 0u;
  if (blockIdx.x == 0u) {
    for (uint32_t i = threadIdx.x; i < a.n; i += blockDim.x) {
      SlabDev q = a.src[i];
      derive(q);
      a.dst[i] = q;
    }
    if (threadIdx.x == 0) *a.ticket = 0ull;
    if (a.bins)
      for (uint32_t i = threadIdx.x; i < a.n * MC_NCOUNT; i += blockDim.x) a.counts[i] = 0ull;
    __syncthreads();
    chain_records(a.dst, a.n, a.order, a.order_begin);
    return;
  }
  if (blockIdx.x <= tblocks) {
    SlabDev q = a.src[blockIdx.x - 1u];
    derive(q);
    write_tables(q, a.tables);
    return;
  }
  const uint64_t nz = (uint64_t)(gridDim.x - 1u - tblocks) * blockDim.x;
  for (uint64_t i = (uint64_t)(blockIdx.x - 1u - tblocks) * blockDim.x + threadIdx.x; i < a.n_slots; i += nz)
    a.bins[i] = 0ull;
}

struct RunArgs {
  const SlabDev* probs;
  uint32_t nprob;
  uint32_t chunk;
  uint64_t range_begin, total;
  unsigned long long* ticket;
  unsigned long long* tally;
  unsigned long long* counts;
  uint64_t* hist_state;
  uint64_t* hist_draws;
  mcd::Lcg lcg;
  uint64_t event_cap;
  uint32_t smem_slots;
  uint32_t smem_edges;  // single-problem launches: n_bins + 1 edges in shared memory (0: none)
  const double* tables; // else per-problem edge and width tables in global memory (nullable)
  uint32_t grab_shift;  // a warp takes at most 2^-grab_shift of the histories left at once,
  uint32_t min_grab;    // but at least min_grab
  uint32_t row_bins;    // bins of a warp's row cache (0: none; all problems fit it otherwise)
  uint32_t walk_pieces; // of a flight's tally a lane adds per pass, after the first
  uint32_t coop_hist;   // histories the block's cooperative tail takes over (0: none)
  uint32_t coop_slots;  // its event records, a power of two
  uint32_t coop_after;  // passes of a warp after the ticket ran out before it offers its histories
  mcs::Order order;        // processing order of several problems (empty: id order)
  mcd::Pow2Maps pow2;
};

// What the end of a history and the cooperative tail need of the launch.
struct TailArgs {
  uint64_t* hist_state;
  uint64_t* hist_draws;
  unsigned long long* counts;
  mcd::Lcg lcg;
  uint64_t event_cap;
};

// The cooperative tail's view of the launch.
struct CoopArgs {
  TailArgs t;
  const SlabDev* probs;
};

// All counts of one ended history, straight to its problem's counters (but
// for its source).
__device__ __noinline__ void count_history(unsigned long long* c, uint64_t events, uint64_t draws, int outcome,
                                           uint64_t stride_q) {
  const bool leaked = outcome == mcs::kLeakLo || outcome == mcs::kLeakHi;
  atomicAdd(c + MC_C_FLIGHTS, (unsigned long long)events);
  atomicAdd(c + MC_C_COLLISIONS, (unsigned long long)(events - (leaked ? 1u : 0u)));
  atomicAdd(c + MC_C_SCATTERS, (unsigned long long)(events - (leaked || outcome == mcs::kAbsorbed ? 1u : 0u)));
  atomicAdd(c + (outcome == mcs::kAbsorbed ? MC_C_ABSORPTIONS : outcome == mcs::kLeakLo ? MC_C_LEAK_LO
                 : outcome == mcs::kLeakHi ? MC_C_LEAK_HI : MC_C_CAPPED), 1ull);
  atomicAdd(c + MC_C_DRAWS, (unsigned long long)draws);
  atomicMax(c + MC_C_MAX_DRAWS, (unsigned long long)draws);
  if (stride_q != 0 && draws > stride_q) {
    atomicAdd(c + MC_C_EXCEED_HIST, 1ull);
    atomicAdd(c + MC_C_EXCEED_DRAWS, (unsigned long long)(draws - stride_q));
  }
}

// A lane's counts for its current problem, few enough to stay in registers
// beside the particle: how many histories started and how they ended, and
// their flights.  Collisions, scatterings and draws follow from these (every
// flight but a leaking one collides, every collision but an absorbing one
// scatters; three draws per event, slab_draws).  Histories that the sums do
// not fit (capped ones, 2^30 flights or more) are counted straight away, and
// exceedances in the block's shared memory (one problem) or straight away.  Flushed with atomics, lane by lane or summed over a
// converged warp first: a problem's counters share a cache line.
struct HistCounts {
  int prob;
  uint32_t src, flights, absn, llo, lhi, maxd;
  __device__ void clear() { src = flights = absn = llo = lhi = maxd = 0u; }
  __device__ static void add(unsigned long long* c, const SlabDev& p, unsigned long long so, unsigned long long fl,
                             unsigned long long ab, unsigned long long lo, unsigned long long hi,
                             unsigned long long mx) {
    const unsigned long long lk = lo + hi, co = fl - lk;
    if (so) atomicAdd(c + MC_C_SOURCE, so);
    if (fl == 0ull) return;  // no history ended
    atomicAdd(c + MC_C_FLIGHTS, fl);
    if (co) atomicAdd(c + MC_C_COLLISIONS, co);
    if (ab) atomicAdd(c + MC_C_ABSORPTIONS, ab);
    if (co != ab) atomicAdd(c + MC_C_SCATTERS, co - ab);
    if (lo) atomicAdd(c + MC_C_LEAK_LO, lo);
    if (hi) atomicAdd(c + MC_C_LEAK_HI, hi);
    atomicAdd(c + MC_C_DRAWS, 3ull * fl - 2ull * lk - ab + (p.source == MC_SRC_BEAM ? 0ull : 2ull * (lk + ab)));
    atomicMax(c + MC_C_MAX_DRAWS, mx);
  }
  __device__ void flush(unsigned long long* counts, const SlabDev* probs) {
    if (prob < 0) return;
    add(counts + (size_t)prob * MC_NCOUNT, probs[prob], src, flights, absn, llo, lhi, maxd);
    clear();
  }
  __device__ void flush_warp(unsigned long long* counts, const SlabDev* probs) {
    const int p = mcd::warp_common_prob(prob);
    if (p == -2) { flush(counts, probs); return; }
    if (p < 0) return;
    const unsigned long long so = mcd::warp_sum64(src), fl = mcd::warp_sum64(flights), ab = mcd::warp_sum64(absn),
                             lo = mcd::warp_sum64(llo), hi = mcd::warp_sum64(lhi), mx = mcd::warp_max64(maxd);
    if ((threadIdx.x & 31u) == 0u) add(counts + (size_t)p * MC_NCOUNT, probs[p], so, fl, ab, lo, hi, mx);
    clear();
  }
};

// End of a history after `events` flights: its counts, its final state and
// draw count where the caller asked for them.  exceed: the block's
// exceedance counts (nullptr: straight to the problem's).
__device__ __forceinline__ void end_history(const TailArgs& t, const SlabDev* probs, uint64_t x, const SlabDev& p,
                                            uint64_t gi, uint64_t events, int outcome, unsigned long long* exceed,
                                            HistCounts& lc) {
  const uint64_t draws = mcs::slab_draws(p, events, outcome);
  if (t.hist_state) t.hist_state[gi] = x & t.lcg.mask;
  if (t.hist_draws) t.hist_draws[gi] = draws;
  unsigned long long* const c = t.counts + (size_t)lc.prob * MC_NCOUNT;
  if (outcome < 0 || events >= (1ull << 30)) {
    count_history(c, events, draws, outcome, p.stride_q);
    return;
  }
  if (p.stride_q != 0 && draws > p.stride_q) {
    atomicAdd(exceed ? exceed : c + MC_C_EXCEED_HIST, 1ull);
    atomicAdd(exceed ? exceed + 1 : c + MC_C_EXCEED_DRAWS, (unsigned long long)(draws - p.stride_q));
  }
  lc.flights += (uint32_t)events;
  lc.absn += outcome == mcs::kAbsorbed ? 1u : 0u;
  lc.llo += outcome == mcs::kLeakLo ? 1u : 0u;
  lc.lhi += outcome == mcs::kLeakHi ? 1u : 0u;
  lc.maxd = max(lc.maxd, (uint32_t)draws);  // below 3 * 2^30 + 2
  if (lc.flights > (1u << 30)) lc.flush(t.counts, probs);
}

// Cooperative tail.  Once the ticket has run out, a block's lanes are no
// longer refilled: what is left is a heavy tail of long histories, and one
// lane runs each of them at the latency of a flight's dependent instructions
// (3600 cycles) while the rest of the block idles.  But a history's draws have
// fixed roles -- each event takes one draw for the distance, one for the
// absorption test and one for the new direction, until the history ends --
// so everything that depends on the draws alone can be computed ahead, by any
// thread.  When a block's live histories are down to a quarter of its threads
// (and have shown that they are long ones), its warps put them into records in
// shared memory and the whole block advances all of them by rounds of E
// events:
//   1. every thread computes events of the round: the product p_e = d_e mu_e,
//      the absorption test and the tally weight, jumping the history's stream
//      to draw 3e with the maps of 2^j steps;
//   2. one thread per history runs the chain of positions alone,
//      x_{e+1} = x_e + p_e and the face tests, until the round ends or the
//      history does (an event cap, a leak, an absorption);
//   3. every thread tallies events of the round.
// E grows as histories end, so that a round always fills the block.  Every
// value comes from the same function, with the same operands, as in the
// one-lane path, so the draws, tallies and counters are the same bits.
//
// An event's record is two words.  fp64: p_e, which the walk replaces by
// x_{e+1}, and the tally weight with the absorption test in its sign bit.
// fp32: the pair (pr, pe), replaced by the position pair, and (wf, muf) with
// the test in wf's sign bit.
constexpr int kCoopHistWords = 14;    // 8-byte words per history record
constexpr int kCoopWords = 2;         // per event record
constexpr int kCoopMaxLog = 8;        // at most 2^8 records per history and round
constexpr int kCoopMinLog = 3;        // at least 2^3: E = 7 events
constexpr uint32_t kCoopMaxHist = 256;

__device__ __forceinline__ mcd::Affine affine_steps(const mcd::Affine* tab, uint64_t k) {
  mcd::Affine acc{1ull, 0ull};
  while (k) {
    const int j = __ffsll((long long)k) - 1;
    acc = mcd::compose(tab[j], acc);
    k &= k - 1;
  }
  return acc;
}

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  return ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
}
__device__ __forceinline__ float lo_of(unsigned long long w) { return __uint_as_float((uint32_t)w); }
__device__ __forceinline__ float hi_of(unsigned long long w) { return __uint_as_float((uint32_t)(w >> 32)); }
__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ double dval(unsigned long long w) { return __longlong_as_double((long long)w); }

// A history's record: its stream, particle, ids and tally sink, and the last
// round it ran.
struct CoopHist {
  unsigned long long* w;
  enum {
    kX = 0,      // stream state
    kPos,        // fp64 x (fp32: xf, xlo)
    kDir,        // fp64 mu (fp32: muf in the high half)
    kW,          // fp64 2^32 / |mu| (fp32: wf in the low half)
    kGi,         // global history index
    kEvents,     // flights flown
    kProb,       // problem index; bit 32: live
    kBase,       // tally row
    kEdges,      // edge and width tables (null: computed)
    kWidths,
    kEnd,        // last round: events run (low half) and how the last one ended (high half)
    kX0,         // stream state and position at its start
    kPos0
  };
  __device__ __forceinline__ explicit CoopHist(unsigned long long* p) : w(p) {}
  __device__ __forceinline__ bool live() const { return (w[kProb] >> 32) != 0ull; }
  __device__ __forceinline__ const SlabDev* prob(const SlabDev* probs) const { return probs + (uint32_t)w[kProb]; }
  __device__ __forceinline__ mcs::Sink sink(bool agg) const {
    return mcs::Sink{reinterpret_cast<unsigned long long*>(w[kBase]), reinterpret_cast<const double*>(w[kEdges]),
                     reinterpret_cast<const double*>(w[kWidths]), agg};
  }
};

constexpr unsigned long long kAbsBit = 1ull << 63;  // fp64 weight word: the event's absorption test

// Phase 1 for event e of E of the history in H, whose stream is xs after the
// 3e draws before it: the event's record, or (e = E) the direction after the
// round.
template <int M, bool F32>
__device__ __forceinline__ void coop_draw(const CoopHist& H, const SlabDev& p, const mcd::Lcg& l, uint64_t xs,
                                          uint32_t e, uint32_t E, unsigned long long* rec) {
  const uint64_t sd = mcd::lcg_step(xs, l.g, l.c);
  const bool absorbed = mcd::u53<M>(mcd::lcg_step(sd, l.g, l.c), l.m) < p.p_abs_n;
  mcs::SlabParticle q;
  mcs::set_direction<F32>(q, mcd::u53<M>(xs, l.m));
  if constexpr (!F32) {
    const double d = __dmul_rn(mclog::neglog1m_n(mcd::u53<M>(sd, l.m)), p.inv_st);
    const double mu = e == 0u ? dval(H.w[CoopHist::kDir]) : q.mu, w = e == 0u ? dval(H.w[CoopHist::kW]) : q.w_mu;
    rec[0] = dbits(e == E ? mu : __dmul_rn(d, mu));
    rec[1] = dbits(w) | (absorbed && e != E ? kAbsBit : 0ull);
  } else {
    const float d = mcs::flight_f32(mcd::u53<M>(sd, l.m)) * p.inv_st_f;
    const float muf = e == 0u ? hi_of(H.w[CoopHist::kDir]) : q.muf, wf = e == 0u ? lo_of(H.w[CoopHist::kW]) : q.wf;
    const float pr = __fmul_rn(d, muf);
    rec[0] = pack2(pr, __fmaf_rn(d, muf, -pr));
    rec[1] = pack2(__uint_as_float(__float_as_uint(wf) | (absorbed && e != E ? 0x80000000u : 0u)), muf);
  }
}

// Phase 2, on one thread: the chain of positions through the round's events,
// until the round ends (kContinue), an event would pass the cap (-1), or the
// history leaks or is absorbed.  Then the history's record moves on by the
// events run, and a history that ended is counted and written out.
template <int M, bool F32>
__device__ __noinline__ void coop_walk(const CoopArgs* c, const mcd::Affine* tab, unsigned long long* hist,
                                       unsigned long long* rec, uint32_t E) {
  const CoopHist H(hist);
  const SlabDev& p = *H.prob(c->probs);
  const uint64_t events = H.w[CoopHist::kEvents], x0 = H.w[CoopHist::kX];
  const uint64_t cap_left = c->t.event_cap - events;  // events never pass the cap
  const uint32_t ok = cap_left < E ? (uint32_t)cap_left : E;
  int out = mcs::kContinue;
  uint32_t e = 0;
  H.w[CoopHist::kX0] = x0;
  H.w[CoopHist::kPos0] = H.w[CoopHist::kPos];
  // Four events at a time while none of them can end the history (no
  // leak, no absorption, no cap, and in fp32 no guard band): the chain of
  // additions runs back to back and one branch takes the four.  Otherwise
  // one event at a time, with the same operations.  (p_e = d_e mu_e has the
  // sign of mu_e, or is zero: the face tests take it for mu_e.)
  if constexpr (!F32) {
    double x = dval(H.w[CoopHist::kPos]);
    const double L = p.L;
    auto leaves = [&](unsigned long long pb, double xn) {
      return ((long long)pb > 0 && !mcs::nn_lt(xn, L)) || ((long long)pb < 0 && __double_as_longlong(xn) <= 0);
    };
    for (;;) {
      unsigned long long* const r = rec + kCoopWords * e;
      if (e + 4u <= ok) {
        const unsigned long long b0 = r[0], b1 = r[2], b2 = r[4], b3 = r[6];
        const unsigned long long a = r[1] | r[3] | r[5] | r[7];
        const double x1 = __dadd_rn(x, dval(b0)), x2 = __dadd_rn(x1, dval(b1)), x3 = __dadd_rn(x2, dval(b2)),
                     x4 = __dadd_rn(x3, dval(b3));
        if (!((a & kAbsBit) != 0ull || leaves(b0, x1) || leaves(b1, x2) || leaves(b2, x3) || leaves(b3, x4))) {
          r[0] = dbits(x1);
          r[2] = dbits(x2);
          r[4] = dbits(x3);
          r[6] = dbits(x4);
          x = x4;
          e += 4u;
          continue;
        }
      }
      if (e == E) break;
      if (e == ok) { out = -1; break; }
      double xn;
      const int f = mcs::advance64(p, x, dval(r[0]), dval(r[0]), xn);
      if (f != mcs::kCollide) { out = f; ++e; break; }
      x = xn;
      r[0] = dbits(x);
      ++e;
      if (r[1] & kAbsBit) { out = mcs::kAbsorbed; break; }
    }
    H.w[CoopHist::kPos] = dbits(x);
    if (out == mcs::kContinue) {
      H.w[CoopHist::kDir] = rec[kCoopWords * E];
      H.w[CoopHist::kW] = rec[kCoopWords * E + 1u];
    }
  } else {
    const unsigned long long pos = H.w[CoopHist::kPos];
    float xf = lo_of(pos), xlo = hi_of(pos);
    const mcd::Lcg l = c->t.lcg;
    for (;;) {
      unsigned long long* const r = rec + kCoopWords * e;
      if (e + 4u <= ok) {
        const unsigned long long q0 = r[0], q1 = r[2], q2 = r[4], q3 = r[6];
        const unsigned long long w0 = r[1], w1 = r[3], w2 = r[5], w3 = r[7];
        float h1, l1, h2, l2, h3, l3, h4, l4;
        mcs::pair_step(xf, xlo, lo_of(q0), hi_of(q0), h1, l1);
        mcs::pair_step(h1, l1, lo_of(q1), hi_of(q1), h2, l2);
        mcs::pair_step(h2, l2, lo_of(q2), hi_of(q2), h3, l3);
        mcs::pair_step(h3, l3, lo_of(q3), hi_of(q3), h4, l4);
        if (((w0 | w1 | w2 | w3) & 0x80000000ull) == 0ull && mcs::plain_collision32(p, hi_of(w0), h1, l1) &&
            mcs::plain_collision32(p, hi_of(w1), h2, l2) && mcs::plain_collision32(p, hi_of(w2), h3, l3) &&
            mcs::plain_collision32(p, hi_of(w3), h4, l4)) {
          r[0] = pack2(h1, l1);
          r[2] = pack2(h2, l2);
          r[4] = pack2(h3, l3);
          r[6] = pack2(h4, l4);
          xf = h4;
          xlo = l4;
          e += 4u;
          continue;
        }
      }
      if (e == E) break;
      if (e == ok) { out = -1; break; }
      float xn, xnlo;
      const int f = mcs::advance32(p, xf, xlo, hi_of(r[1]), lo_of(r[0]), hi_of(r[0]),
                                   [&] { return mcd::u53<M>(mcs::skip_tab(tab, x0, 3ull * e + 1ull), l.m); }, xn, xnlo);
      if (f != mcs::kCollide) { out = f; ++e; break; }
      xf = xn;
      xlo = xnlo;
      r[0] = pack2(xf, xlo);
      ++e;
      if (r[1] & 0x80000000ull) { out = mcs::kAbsorbed; break; }
    }
    H.w[CoopHist::kPos] = pack2(xf, xlo);
    if (out == mcs::kContinue) {
      H.w[CoopHist::kDir] = rec[kCoopWords * E + 1u];
      H.w[CoopHist::kW] = rec[kCoopWords * E + 1u];
    }
  }
  const uint64_t total = events + e;
  H.w[CoopHist::kEvents] = total;
  H.w[CoopHist::kEnd] = (unsigned long long)e | ((unsigned long long)(uint32_t)out << 32);
  // draws the round took: three per completed event, one for a leaking
  // flight, two for an absorbed one, none for a capped event
  const uint64_t used = out == mcs::kContinue ? 3ull * E
                      : out == -1 ? 3ull * e
                      : out == mcs::kAbsorbed ? 3ull * e - 1ull : 3ull * e - 2ull;
  const uint64_t x = mcs::skip_tab(tab, x0, used);
  H.w[CoopHist::kX] = x;
  if (out == mcs::kContinue) return;
  // the history's end
  const uint64_t draws = mcs::slab_draws(p, total, out);
  const uint32_t pi = (uint32_t)H.w[CoopHist::kProb];
  count_history(c->t.counts + (size_t)pi * MC_NCOUNT, total, draws, out, p.stride_q);
  const uint64_t gi = H.w[CoopHist::kGi];
  if (c->t.hist_state) c->t.hist_state[gi] = x & c->t.lcg.mask;
  if (c->t.hist_draws) c->t.hist_draws[gi] = draws;
  H.w[CoopHist::kProb] = pi;  // no longer live
}

// Phase 3 for event e of those the history in H ran (nev, the last one
// ending as out): its tally, from its positions x_e and x_{e+1}.  With
// warp-aggregated atomics whatever the launch's setting (the bits are the
// same either way): neighbouring threads tally neighbouring events of one
// history, mostly in the same bins.  A direction of exactly zero (weight 0)
// needs the flight's distance, drawn again.
template <int M, bool F32>
__device__ __forceinline__ void coop_tally(const CoopHist& H, const SlabDev& p, const mcd::Lcg& l,
                                           const mcd::Affine* tab, uint32_t e, uint32_t nev, int out,
                                           const unsigned long long* rec) {
  const mcs::Sink sk = H.sink(true);
  const int f = e == nev - 1u && (out == mcs::kLeakLo || out == mcs::kLeakHi) ? out : mcs::kCollide;
  const unsigned long long from = e == 0u ? H.w[CoopHist::kPos0] : rec[-kCoopWords];
  auto n_dist = [&] { return mcd::u53<M>(mcs::skip_tab(tab, H.w[CoopHist::kX0], 3ull * e + 1ull), l.m); };
  if constexpr (!F32) {
    const double x = dval(from), w = dval(rec[1] & ~kAbsBit);
    int j = mcs::bin_of(p, sk, x);
    if (f == mcs::kCollide && mcx::d_zero(w)) {
      sk.add(j, mcx::fix32_nonneg(__dmul_rn(mclog::neglog1m_n(n_dist()), p.inv_st)));
      return;
    }
    const double xe = f == mcs::kLeakHi ? p.L : (f == mcs::kLeakLo ? 0.0 : dval(rec[0]));
    const mcs::Walk64<true> k{xe, w, !mcs::nn_lt(xe, x)};
    if (mcs::walk_first(p, x, k, sk, j))
      while (mcs::walk_next(p, k, sk, j)) {}
  } else {
    const unsigned long long to = rec[0];
    const float xf = lo_of(from), xlo = hi_of(from), muf = hi_of(rec[1]);
    const float wf = __uint_as_float((uint32_t)rec[1] & 0x7fffffffu);
    int j = mcs::bin_of_pair(p, xf, xlo);
    const float d = muf == 0.0f ? mcs::flight_f32(n_dist()) * p.inv_st_f : 0.0f;  // (used for a zero direction alone)
    mcs::tally32(p, xf, xlo, lo_of(to), hi_of(to), muf, d, wf, f, sk, j);
  }
}

// The rounds, by the whole block, over the n history records at hist, with
// `slots` event records after them.
template <int M, bool F32>
__device__ __noinline__ void coop_tail(const CoopArgs* c, const mcd::Affine* tab, unsigned long long* hist,
                                       unsigned long long* recs, uint32_t slots, uint32_t n) {
  __shared__ uint16_t s_list[kCoopMaxHist];  // the live histories' records
  __shared__ uint32_t s_live;
  const uint32_t t = threadIdx.x, T = blockDim.x;
  __syncthreads();  // the arguments are in place
  const mcd::Lcg l = c->t.lcg;
  uint32_t map_e = ~0u;
  mcd::Affine map{1ull, 0ull};
  for (;;) {
    __syncthreads();
    if (t < 32u) {
      uint32_t cnt = 0;
      for (uint32_t b = 0; b < n; b += 32u) {
        const bool live = b + t < n && CoopHist(hist + (size_t)(b + t) * kCoopHistWords).live();
        const unsigned m = __ballot_sync(0xffffffffu, live);
        if (live) s_list[cnt + __popc(m & ((1u << t) - 1u))] = (uint16_t)(b + t);
        cnt += __popc(m);
      }
      if (t == 0u) s_live = cnt;
    }
    __syncthreads();
    const uint32_t H = s_live;
    if (H == 0u) break;
    int k = kCoopMaxLog;
    while (k > kCoopMinLog && (H << k) > slots) --k;
    const uint32_t S = 1u << k, E = S - 1u;
    for (uint32_t s = t; s < H << k; s += T) {
      const uint32_t e = s & (S - 1u);
      if (e != map_e) {  // (the same for all of a thread's events when S divides the block)
        map = affine_steps(tab, 3ull * e);
        map_e = e;
      }
      const CoopHist h(hist + (size_t)s_list[s >> k] * kCoopHistWords);
      coop_draw<M, F32>(h, *h.prob(c->probs), l, mcd::apply(map, h.w[CoopHist::kX]), e, E, recs + (size_t)kCoopWords * s);
    }
    __syncthreads();
    for (uint32_t i = t; i < H; i += T)
      coop_walk<M, F32>(c, tab, hist + (size_t)s_list[i] * kCoopHistWords, recs + ((size_t)kCoopWords * i << k), E);
    __syncthreads();
    for (uint32_t s = t; s < H << k; s += T) {
      const CoopHist h(hist + (size_t)s_list[s >> k] * kCoopHistWords);
      const uint32_t e = s & (S - 1u), nev = (uint32_t)h.w[CoopHist::kEnd];
      if (e < nev)
        coop_tally<M, F32>(h, *h.prob(c->probs), l, tab, e, nev, (int)(uint32_t)(h.w[CoopHist::kEnd] >> 32),
                           recs + (size_t)kCoopWords * s);
    }
  }
}

constexpr uint32_t kMaxRowBins = 256;  // of a warp's row cache (2 KiB)

// Lane-passes of waiting after which a warp refills (8 to 32 measure within 2 %
// of each other; refilling at every pass that finds a dead lane: 256 problems
// fp32 10.9 ms against 10.6, fp64 17.3 against 15.0).
constexpr uint32_t kIdle = 16;

// Lanes still walking for which a warp adds another piece of its tallies in
// the same pass.  A tally in shared memory is a single problem's, or small:
// one lane, and slab_walk_pieces the limit (with 8 lanes 300 000 histories of 9
// flights took 260 us instead of 253).  Otherwise problems of many kinds share
// the warps and no number of pieces suits all: no limit but 8 lanes (256
// problems, against two pieces: fp32 8.72 -> 8.55 ms, fp64 13.1 -> 12.4 ms; 4,
// 6 and 12 lanes within 2 %).
template <bool SMEM> constexpr int kWalkMin = SMEM ? 1 : 8;
// Once the work has run out, all lanes that are left are enough as well: while
// every one of them walks, none waits for the next pass.  Blocks of one warp
// run so for long, without a cooperative tail (5000 histories at 100 bins per
// mean free path: 1.91 s with a pass for each piece then, 1.21 now; 1.54
// before passes were split, 1.25 going on for half of the lanes).  The kernel
// of small runs has the registers for it; those of 64 and 80 do without, whose
// long histories go to the tail (there it cost 256 problems 1 %: 8.54 -> 8.63
// ms), but for generic widths and warp-aggregated tallies, which have no other.
template <int M, bool SMEM, bool AGG, bool FEW> constexpr bool kWalkLast = !SMEM && (FEW || M != 63 || AGG);
constexpr uint32_t kWalkNoLimit = ~0u;

// The ticket positions of one problem: begin + id for its history id.
struct Span {
  uint64_t begin;
  uint32_t prob;
};

// Adds a warp's row cache to its tally row in global memory and clears it.
__device__ __forceinline__ void flush_row(unsigned long long* global_row, uint32_t row, uint32_t n_bins) {
  extern __shared__ unsigned long long s_dyn[];
  __syncwarp();
  for (uint32_t j = threadIdx.x & 31u; j < n_bins; j += 32u) {
    const unsigned long long v = s_dyn[row + j];
    if (v == 0ull) continue;
    s_dyn[row + j] = 0ull;
    atomicAdd(global_row + j, v);
  }
  __syncwarp();
}

template <int M, bool F32, bool SMEM, bool AGG, bool FEW>
__device__ __forceinline__ void slab_history_body(const RunArgs& a) {
  constexpr bool LAST = kWalkLast<M, SMEM, AGG, FEW>;
  extern __shared__ unsigned long long s_dyn[];
  unsigned long long* const s_tally = s_dyn;
  __shared__ mcd::Affine tab[64];
  mcd::load_maps(a.pow2, tab);
  if constexpr (SMEM) {
    for (uint32_t s = threadIdx.x; s < a.smem_slots; s += blockDim.x) s_tally[s] = 0ull;
  }
  double* s_edges = a.smem_edges ? reinterpret_cast<double*>(s_tally + (SMEM ? a.smem_slots : 0u)) : nullptr;
  double* s_widths = s_edges ? s_edges + a.smem_edges : nullptr;  // n_bins widths after the edges
  // the cooperative tail's records after the tally and the edge tables
  unsigned long long* s_coop = s_tally + (SMEM ? a.smem_slots : 0u) + 2u * a.smem_edges;
  __shared__ uint32_t s_live[16];   // per warp: an upper bound on its live histories
  __shared__ uint32_t s_go, s_n;    // the tail has begun; histories in its records
  __shared__ unsigned long long s_exceed[2];  // one problem: exceeding histories, and their draws beyond Q
  if (threadIdx.x == 0) {
    s_exceed[0] = s_exceed[1] = 0ull;
    s_go = s_n = 0u;
  }
  // the warps' row caches after those
  const uint32_t row0 = (SMEM ? a.smem_slots : 0u) + 2u * a.smem_edges + a.coop_hist * kCoopHistWords + a.coop_slots * kCoopWords;
  if constexpr (!SMEM)
    for (uint32_t i = threadIdx.x; i < (blockDim.x >> 5) * a.row_bins; i += blockDim.x) s_dyn[row0 + i] = 0ull;
  __shared__ Span s_span[16];
  if (threadIdx.x < 16u) s_span[threadIdx.x] = Span{1ull << 63, 0u};
  if (threadIdx.x < 16u) s_live[threadIdx.x] = threadIdx.x < (blockDim.x >> 5) ? kCoopMaxHist : 0u;
  if (s_edges) {
    const SlabDev& p0 = a.probs[0];
    for (uint32_t j = threadIdx.x; j + 1 < a.smem_edges; j += blockDim.x)
      s_widths[j] = __dsub_rn(mcs::slab_edge(p0, (int)j + 1), mcs::slab_edge(p0, (int)j));
  }
  if (s_edges) {
    const SlabDev& p0 = a.probs[0];
    for (uint32_t j = threadIdx.x; j < a.smem_edges; j += blockDim.x) s_edges[j] = mcs::slab_edge(p0, (int)j);
  }
  __syncthreads();

  const unsigned kFull = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;
  const mcd::Lcg l = a.lcg;

  uint64_t pool_next = 0, pool_end = 0;
  uint32_t grab = a.chunk, idle = 0;
  bool more = true;
  bool alive = false;
  HistCounts lc;
  lc.prob = -1;
  lc.clear();

  const SlabDev* P = a.probs;
  uint64_t x = 0;  // stream state
  mcs::SlabParticle q{};
  mcs::Sink sink{nullptr, s_edges, s_widths, AGG};
  uint64_t gi = 0, events = 0;
  typename mcs::WalkOf<F32>::type wk{};  // the rest of the current flight's tally, while `walking`
  bool walking = false;
  int outcome = mcs::kContinue;          // of the history's last event
  uint32_t after = 0;  // passes since the ticket ran out
  const uint32_t my_row = row0 + (threadIdx.x >> 5) * a.row_bins;
  unsigned long long* row_of = nullptr;  // the tally row the warp's cache accumulates
  uint32_t row_n = 0;                    // its bins

  for (;;) {
    unsigned dead = __ballot_sync(kFull, !alive);
    const unsigned waiting = dead;
    // A refill (seed, source draws, the problem's lookup) costs the warp the
    // same for one lane as for many, about what kIdle lanes lose by waiting
    // a pass.
    idle += (uint32_t)__popc(dead);
    const bool refill = idle >= kIdle || dead == kFull;
    if (refill) idle = 0u;
    while (refill && dead != 0u && more) {
      if (pool_next >= pool_end) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(a.ticket, (unsigned long long)grab);
        base = __shfl_sync(kFull, base, 0);
        if (base >= a.total) { more = false; break; }
        pool_next = base;
        pool_end = min((uint64_t)base + (uint64_t)grab, (uint64_t)a.total);
        // smaller chunks towards the end, so that the warps run out together
        grab = (uint32_t)min((uint64_t)a.chunk, max((uint64_t)a.min_grab, (a.total - pool_next) >> a.grab_shift));
      }
      const uint64_t avail = pool_end - pool_next;
      const unsigned rank = __popc(dead & lt_mask);
      if (!alive && rank < avail) {
        uint32_t pi = 0;
        const uint64_t t = pool_next + rank;
        uint64_t id = 0;
        if (a.nprob != 1u) {  // mostly the problem the warp's last history was of
          pi = s_span[threadIdx.x >> 5].prob;
          id = t - s_span[threadIdx.x >> 5].begin;
        }
        if (a.nprob == 1u || id >= a.probs[pi].n_hist) {
          mcs::ticket_history(a.probs, a.nprob, a.range_begin, a.order, t, pi, gi);
          id = gi - a.probs[pi].hist_begin;
        }
        if ((int)pi != lc.prob) { lc.flush(a.counts, a.probs); lc.prob = (int)pi; }
        P = a.probs + pi;
        gi = P->hist_begin + id;
        const uint64_t batch = P->n_batches > 1u ? mcs::batch_of(id, P->n_hist, P->n_batches) : 0ull;
        sink.base = (SMEM ? s_tally : a.tally) + P->tally_offset + batch * P->n_bins;
        if (a.tables) {
          sink.edges = a.tables + P->tab_off;
          sink.widths = sink.edges + P->n_bins + 1;
        }
        mcs::Rng<M> r{mcs::slab_seed(*P, id, tab, l.mask), 0ull};
        mcs::slab_source<M, F32>(*P, r, l, q);
        x = r.x;
        q.j = mcs::locate<F32>(*P, q, sink);
        events = 0;
        outcome = mcs::kContinue;
        ++lc.src;
        alive = true;
      }
      if (a.nprob != 1u) {  // the last position taken: its problem's span of positions
        __syncwarp();
        if ((dead & (1u << lane)) != 0u && rank + 1u == min((uint64_t)__popc(dead), avail))
          s_span[threadIdx.x >> 5] = Span{pool_next + rank - (gi - P->hist_begin), (uint32_t)(P - a.probs)};
        __syncwarp();
      }
      pool_next += min((uint64_t)__popc(dead), avail);
      dead = __ballot_sync(kFull, !alive);
    }
    if (!SMEM && a.row_bins != 0u && dead != waiting) {
      // new histories: the row most lanes are on is the one the warp caches
      if (waiting & (1u << lane)) sink.row = mcs::kNoRow;
      unsigned out = __ballot_sync(kFull, alive && sink.base != row_of) & waiting;
      if (out != 0u) {
        const int who = 31 - __clz((int)out);
        unsigned long long* const cand = reinterpret_cast<unsigned long long*>(
            __shfl_sync(kFull, reinterpret_cast<unsigned long long>(sink.base), who));
        const uint32_t n = __shfl_sync(kFull, alive ? P->n_bins : 0u, who);
        if (__popc(__ballot_sync(kFull, alive && sink.base == cand)) >
            __popc(__ballot_sync(kFull, alive && sink.base == row_of))) {
          if (row_of) flush_row(row_of, my_row, row_n);
          row_of = cand;
          row_n = n;
        }
      }
      sink.row = alive && sink.base == row_of ? my_row : mcs::kNoRow;
    }
    if (dead == kFull) {
      if (lane == 0) s_live[threadIdx.x >> 5] = 0u;
      break;
    }
    if (!more && a.coop_hist != 0u && ++after >= a.coop_after) {
      // The block's live histories, from each warp's own count (a warp that
      // still refills, or has not run coop_after passes since, counts as
      // full).  Counts only fall, so a sum read while they change is an upper
      // bound, and whoever finds it small enough starts the tail for all.
      volatile uint32_t* const vl = s_live;
      if (lane == 0) vl[threadIdx.x >> 5] = (uint32_t)__popc(~dead);
      const uint32_t mine = lane < 16u ? vl[lane] : 0u;
      const bool go = __reduce_add_sync(kFull, mine) <= a.coop_hist || *(volatile uint32_t*)&s_go != 0u;
      if (__any_sync(kFull, go)) {
        // between two events: tallies under way are completed first, and the
        // histories that they were the end of
        while (walking) walking = mcs::walk_next(*P, wk, sink, q.j);
        if (alive && outcome != mcs::kContinue) {
          end_history(TailArgs{a.hist_state, a.hist_draws, a.counts, a.lcg, a.event_cap}, a.probs, x, *P, gi, events,
                      outcome, a.nprob == 1 ? s_exceed : nullptr, lc);
          alive = false;
        }
        dead = __ballot_sync(kFull, !alive);
        uint32_t base = 0;
        if (lane == 0) {
          *(volatile uint32_t*)&s_go = 1u;
          base = atomicAdd(&s_n, (uint32_t)__popc(~dead));
        }
        base = __shfl_sync(kFull, base, 0);
        const uint32_t at = base + (uint32_t)__popc(~dead & lt_mask);
        if (alive && at < a.coop_hist) {  // always, by the bound
          unsigned long long* const w = s_coop + (size_t)at * kCoopHistWords;
          w[CoopHist::kX] = x;
          w[CoopHist::kPos] = F32 ? pack2(q.xf, q.xlo) : dbits(q.x);
          w[CoopHist::kDir] = F32 ? pack2(0.0f, q.muf) : dbits(q.mu);
          w[CoopHist::kW] = F32 ? pack2(q.wf, 0.0f) : dbits(q.w_mu);
          w[CoopHist::kGi] = gi;
          w[CoopHist::kEvents] = events;
          w[CoopHist::kProb] = (uint64_t)(uint32_t)(P - a.probs) | (1ull << 32);
          w[CoopHist::kBase] = reinterpret_cast<unsigned long long>(sink.base);
          w[CoopHist::kEdges] = reinterpret_cast<unsigned long long>(sink.edges);
          w[CoopHist::kWidths] = reinterpret_cast<unsigned long long>(sink.widths);
        } else if (alive) {
          atomicAdd(a.counts + MC_C_DROPPED, 1ull);
        }
        break;
      }
    }
    if (alive && !walking) {
      outcome = -1;  // event cap
      if (events != a.event_cap) {
        ++events;
        outcome = mcs::slab_event<M, F32>(*P, x, l, q, sink, wk, walking);
      }
    }
    // The other pieces of the tallies, walk_pieces per lane at most and, after
    // the first, only for kWalkMin lanes together (LAST: or all that are left):
    // a lane whose flight crosses more bins goes on in the next pass, while the
    // others take their next event.
    for (uint32_t i = 0; i < a.walk_pieces; ++i) {
      const unsigned on = __ballot_sync(kFull, walking);
      if (__popc(on) < (i == 0u ? 1 : kWalkMin<SMEM>) && (!LAST || more || on == 0u || (on | dead) != kFull)) break;
      if (walking) walking = mcs::walk_next(*P, wk, sink, q.j);
    }
    if (alive && !walking && outcome != mcs::kContinue) {
      end_history(TailArgs{a.hist_state, a.hist_draws, a.counts, a.lcg, a.event_cap}, a.probs, x, *P, gi, events, outcome,
                  a.nprob == 1 ? s_exceed : nullptr, lc);
      alive = false;
    }
  }
  lc.flush_warp(a.counts, a.probs);
  if (!SMEM && row_of) flush_row(row_of, my_row, row_n);

  __syncthreads();
  if (s_n != 0u) {
    // the arguments through shared memory: a call with them by value would
    // put them on the stack of the whole kernel
    __shared__ CoopArgs s_args;
    if (threadIdx.x == 0) s_args = CoopArgs{TailArgs{a.hist_state, a.hist_draws, a.counts, a.lcg, a.event_cap}, a.probs};
    coop_tail<M, F32>(&s_args, tab, s_coop, s_coop + (size_t)a.coop_hist * kCoopHistWords, a.coop_slots,
                      min(s_n, a.coop_hist));
  }
  if (threadIdx.x == 0 && s_exceed[0] != 0ull) {
    atomicAdd(a.counts + MC_C_EXCEED_HIST, s_exceed[0]);
    atomicAdd(a.counts + MC_C_EXCEED_DRAWS, s_exceed[1]);
  }
  if constexpr (SMEM) {
    for (uint32_t s = threadIdx.x; s < a.smem_slots; s += blockDim.x) {
      const unsigned long long v = s_tally[s];
      if (v != 0ull) atomicAdd(a.tally + s, v);
    }
  }
}

// The kernel in two register budgets.  The fp32 flight fits 64 registers but
// for a few spills (four blocks of 256 per SM; at 80, 256 problems took a
// tenth longer); the fp64 flight runs fastest with 80 and three blocks per SM
// (slab_long at 64 / 72 / 80 / 96 registers 166 / 159 / 156 / 180 ms when each was
// tried, before the bin walk was split; 136 ms at 80 as it is).  Both accept
// blocks of up to 512 threads.
template <int M, bool F32, bool SMEM, bool AGG>
__global__ void __launch_bounds__(512, 2) slab_history_kernel_f32(const RunArgs a) {
  slab_history_body<M, F32, SMEM, AGG, false>(a);
}
template <int M, bool F32, bool SMEM, bool AGG>
__global__ void __maxnreg__(80) slab_history_kernel_f64(const RunArgs a) {
  slab_history_body<M, F32, SMEM, AGG, false>(a);
}

// A run of at most a few warps per SM waits for its longest histories, not for
// issue slots: registers to interleave an event's chains are worth more than
// warps that are not there (10^4 histories, fp64: 53 us a call at 96 registers
// and more against 59 at 80; with one launch to set up, 38).
template <int M, bool F32, bool SMEM, bool AGG>
__global__ void __maxnreg__(128) slab_history_kernel_few(const RunArgs a) {
  slab_history_body<M, F32, SMEM, AGG, true>(a);
}

constexpr uint64_t kFewThreads = 128;  // per SM, at most, for the kernel of small runs

template <int M, bool F32, bool SMEM, bool AGG>
auto history_kernel_of(bool few) {
  if constexpr (M == 63 && !AGG) {
    if (few) return slab_history_kernel_few<M, F32, SMEM, AGG>;
  }
  if constexpr (F32) return slab_history_kernel_f32<M, F32, SMEM, AGG>;
  else return slab_history_kernel_f64<M, F32, SMEM, AGG>;
}

template <int M, bool F32, bool SMEM, bool AGG>
int launch_history(const RunArgs& a0, int block, int blocks_per_sm, int num_sms, cudaStream_t s) {
  RunArgs a = a0;
  // Enough warps for every chunk, never more than fill the GPU.
  const uint64_t warps_needed = (a.total + a.chunk - 1) / a.chunk;
  const uint64_t blocks_needed = (warps_needed * 32 + block - 1) / block;
  const bool few = blocks_needed * (uint64_t)block <= (uint64_t)num_sms * kFewThreads;
  auto k = history_kernel_of<M, F32, SMEM, AGG>(few);
  // What the driver says about this kernel on this device, asked for once: its
  // static shared memory, the opt-in limit, and after the request for all of
  // that, the blocks per SM of the last launch shape.
  struct Known {
    int dev = -1, optin = 0, block = 0, per_sm = 0;
    size_t static_smem = 0, smem = 0;
  };
  static thread_local Known known[2];
  Known& kn = known[few ? 1 : 0];
  int dev = 0;
  cudaGetDevice(&dev);
  if (kn.dev != dev) {
    cudaFuncAttributes fa{};
    int st = mci::cuda_status(cudaFuncGetAttributes(&fa, k), "cudaFuncGetAttributes(slab_history_kernel)");
    if (st != MC_OK) return st;
    Known n;
    st = mci::cuda_status(cudaDeviceGetAttribute(&n.optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev),
                          "cudaDeviceGetAttribute(shared memory)");
    if (st != MC_OK) return st;
    n.static_smem = fa.sharedSizeBytes;
    st = mci::cuda_status(
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, n.optin - (int)n.static_smem),
        "cudaFuncSetAttribute(slab_history_kernel)");
    if (st != MC_OK) return st;
    n.dev = dev;
    kn = n;
  }
  const size_t optin = (size_t)kn.optin, static_smem = kn.static_smem;
  // What does not fit beside the static part is given up, the row caches first,
  // then the cooperative tail and the edge tables (all only save time).
  auto dynamic_smem = [&a, block]() {
    return (SMEM ? (size_t)a.smem_slots * 8u : 0u) + (size_t)a.smem_edges * 16u +  // edges + widths
           ((size_t)a.coop_hist * kCoopHistWords + (size_t)a.coop_slots * kCoopWords) * 8u +
           (size_t)(block / 32) * a.row_bins * 8u;
  };
  if (SMEM || a.row_bins > kMaxRowBins) a.row_bins = 0;
  if (static_smem + dynamic_smem() > optin) a.row_bins = 0;
  if (static_smem + dynamic_smem() > optin) a.coop_hist = a.coop_slots = 0;
  if (static_smem + dynamic_smem() > optin) a.smem_edges = 0;
  const size_t smem = dynamic_smem();
  if (static_smem + smem > optin) {
    mci::set_error("slab_history_kernel: %u tally slots do not fit in shared memory", a.smem_slots);
    return MC_ERR_ARG;
  }
  int per_sm = blocks_per_sm;
  if (per_sm <= 0) {
    if (kn.per_sm == 0 || kn.block != block || kn.smem != smem) {
      int st = mci::cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem),
                                "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
      if (st != MC_OK) return st;
      kn.per_sm = std::max(per_sm, 1);
      kn.block = block;
      kn.smem = smem;
    }
    per_sm = kn.per_sm;
  }
  const uint64_t full = (uint64_t)num_sms * (uint64_t)per_sm;
  const int grid = (int)std::max<uint64_t>(1, std::min(full, blocks_needed));
  a.grab_shift = 1u;  // twice the launch's warps, rounded up to a power of two
  while ((1ull << a.grab_shift) < 2ull * (uint64_t)grid * (uint64_t)(block / 32)) ++a.grab_shift;
  k<<<grid, block, smem, s>>>(a);
  return mci::cuda_status(cudaGetLastError(), "slab_history_kernel launch");
}

template <int M, bool AGG>
int launch_history_m(const RunArgs& a, bool f32, int block, int bps, int sms, cudaStream_t s) {
  const bool smem = a.smem_slots != 0;
  if (f32) return smem ? launch_history<M, true, true, AGG>(a, block, bps, sms, s)
                       : launch_history<M, true, false, AGG>(a, block, bps, sms, s);
  return smem ? launch_history<M, false, true, AGG>(a, block, bps, sms, s)
              : launch_history<M, false, false, AGG>(a, block, bps, sms, s);
}

}  // namespace

namespace mci {

size_t slab_dev_size() { return sizeof(SlabDev); }

void slab_fill_host(const mc_problem* src, uint32_t n, void* dst) {
  SlabDev* d = static_cast<SlabDev*>(dst);
  uint64_t off = 0;
  for (uint32_t i = 0; i < n; ++i) {
    SlabDev q;
    std::memset(&q, 0, sizeof q);
    q.L = src[i].L;
    q.sigma_t = src[i].sigma_t;
    q.c = src[i].c;
    q.n_hist = src[i].n_histories;
    q.seed = src[i].seed;
    q.stride_q = src[i].stride_q;
    q.id_offset = src[i].id_offset;
    q.key = src[i].key;
    q.tally_offset = src[i].tally_offset;
    q.n_bins = src[i].n_bins;
    q.n_batches = src[i].n_batches;
    q.source = src[i].source;
    q.seeding = src[i].seeding;
    q.tab_off = off;
    off += 2ull * q.n_bins + 1ull;
    d[i] = q;
  }
}

int slab_prep(void* d_probs, uint32_t n, cudaStream_t s, void* d_tables, void* d_order) {
  uint32_t* order = d_order && n >= 2 && n <= kMaxOrderedProblems ? static_cast<uint32_t*>(d_order) : nullptr;
  uint64_t* begin = order ? reinterpret_cast<uint64_t*>(order + ((n + 1u) & ~1u)) : nullptr;
  slab_prep_kernel<<<1, 256, 0, s>>>(static_cast<SlabDev*>(d_probs), n, order, begin);
  int st = cuda_status(cudaGetLastError(), "slab_prep_kernel launch");
  if (st != MC_OK || !d_tables) return st;
  slab_tables_kernel<<<std::min<uint32_t>(n, 1024u), 64, 0, s>>>(static_cast<const SlabDev*>(d_probs), n,
                                                                   static_cast<double*>(d_tables));
  return cuda_status(cudaGetLastError(), "slab_tables_kernel launch");
}

int slab_init(const void* records, uint32_t n, void* d_probs, void* d_tables, void* d_order, const mc_tally* tally,
              bool zero, unsigned long long* d_ticket, cudaStream_t s) {
  InitArgs a;
  std::memcpy(a.src, records, n * sizeof(SlabDev));
  a.n = n;
  a.dst = static_cast<SlabDev*>(d_probs);
  a.order = n >= 2 ? static_cast<uint32_t*>(d_order) : nullptr;
  a.order_begin = a.order ? reinterpret_cast<uint64_t*>(a.order + ((n + 1u) & ~1u)) : nullptr;
  a.tables = static_cast<double*>(d_tables);
  a.ticket = d_ticket;
  a.bins = zero ? reinterpret_cast<unsigned long long*>(tally->d_bins) : nullptr;
  a.counts = reinterpret_cast<unsigned long long*>(tally->d_counts);
  a.n_slots = zero ? tally->n_slots : 0u;
  const uint32_t zblocks = (uint32_t)std::min<uint64_t>((a.n_slots + 511u) / 512u, 1024u);
  slab_init_kernel<<<1u + (a.tables ? n : 0u) + zblocks, 128, 0, s>>>(a);
  return cuda_status(cudaGetLastError(), "slab_init_kernel launch");
}

uint64_t slab_table_doubles(const mc_problem* src, uint32_t n) {
  uint64_t t = 0;
  for (uint32_t i = 0; i < n; ++i) t += 2ull * src[i].n_bins + 1ull;
  return t;
}

// Pieces per pass of a run whose tally is in shared memory, from the edges an
// average flight crosses, (1/2) bins per mean free path (averaged over the
// histories): as many as most flights need.  slab_long (1/2): 1 / 2 / 3 / all
// of them 141 / 148 / 159 / 163 ms; 300 000 histories of 9 flights (1.1): 264 /
// 257 / 269 us with 1 / 2 / 3.
uint32_t slab_walk_pieces(const mc_problem* src, uint32_t n) {
  double bins = 0.0, paths = 0.0;
  for (uint32_t i = 0; i < n; ++i) {
    bins += (double)src[i].n_histories * src[i].n_bins;
    paths += (double)src[i].n_histories * src[i].L * src[i].sigma_t;
  }
  const double crossed = 0.5 * bins / std::max(paths, 1e-300);
  return crossed < 0.75 ? 1u : crossed < 2.0 ? 2u : crossed < 6.0 ? 3u : 4u;
}

int slab_history_launch(const SlabLaunch& L, cudaStream_t s) {
  RunArgs a{};
  a.probs = static_cast<const SlabDev*>(L.d_probs);
  a.nprob = L.n_problems;
  a.chunk = L.chunk;
  a.range_begin = L.range_begin;
  a.total = L.total;
  a.ticket = L.d_ticket;
  a.tally = reinterpret_cast<unsigned long long*>(L.tally->d_bins);
  a.counts = reinterpret_cast<unsigned long long*>(L.tally->d_counts);
  a.hist_state = L.tally->d_hist_state;
  a.hist_draws = L.tally->d_hist_draws;
  a.lcg = mcd::Lcg{L.lcg.g, L.lcg.c, mcd::mask_of(L.lcg.m), L.lcg.m};
  a.event_cap = L.event_cap;
  a.pow2 = mcd::pow2_maps(L.lcg.g, L.lcg.c);
  a.smem_slots = L.smem_slots;
  a.smem_edges = 0;
  if (L.n_problems == 1) {
    // one problem: its bin edges from a shared-memory table (the problem's
    // bin count comes from the host copy through the launch descriptor)
    if (L.single_n_bins + 1 <= 4096) a.smem_edges = L.single_n_bins + 1;
  }
  // otherwise each problem's tables in global memory, where staged
  a.tables = a.smem_edges ? nullptr : static_cast<const double*>(L.d_tables);
  // One problem: chunks down to 8 histories at the end, so that the warps run
  // out together (300 000 histories of 9 flights: 321 -> 312 us).  Several: a
  // chunk that spans few problems is worth more (256 problems fp32: 11.0 ms
  // with whole chunks, 11.6 with chunks down to 8 or 32).
  a.min_grab = L.n_problems == 1 ? 8u : a.chunk;
  // The cooperative tail takes over when a quarter of a block's threads still
  // carry a history, with four event records per thread in fp64 and two in
  // fp32 (a power of two).  slab_long, 10^6 histories, when each was tried,
  // before the bin walk was split: fp64 154 ms, against 164 with half the threads
  // and 157 with two records; fp32 107 ms, against 114 with four records; without
  // the tail 244 and 160 ms.  (As it is 136 and 107 ms.)  coop_after: passes after
  // which what is left counts as long (16: 298 us instead of 292 for 300 000
  // histories of 9 flights, 4: 329; long chains do not care)
  a.coop_after = 32u;
  if (L.pool_lock_attempts != 0u && L.block >= 64) {
    a.coop_slots = 128u;
    while (a.coop_slots * 2u <= (uint32_t)L.block * (L.f32 ? 2u : 4u)) a.coop_slots *= 2u;
    // (a round's records, at least 2^kCoopMinLog per history, must fit)
    a.coop_hist = std::min((uint32_t)L.block / 4u, a.coop_slots >> kCoopMinLog);
  }
  // Without the whole tally in shared memory each warp accumulates the row
  // most of its lanes are on in a cache of its own: all warps work through the
  // problems in one order, and their atomics met at a few lines of L2 (256
  // problems: fp32 16.6 -> 11.0 ms, fp64 21.2 -> 17.0 ms).
  a.row_bins = L.max_n_bins;
  a.walk_pieces = L.smem_slots != 0u ? L.walk_pieces : kWalkNoLimit;
  a.order = mcs::Order{L.d_order, L.d_order_begin};
  if (L.tally_agg) {
    if (L.lcg.m == 63) return launch_history_m<63, true>(a, L.f32, L.block, L.blocks_per_sm, L.num_sms, s);
    return launch_history_m<0, true>(a, L.f32, L.block, L.blocks_per_sm, L.num_sms, s);
  }
  if (L.lcg.m == 63) return launch_history_m<63, false>(a, L.f32, L.block, L.blocks_per_sm, L.num_sms, s);
  return launch_history_m<0, false>(a, L.f32, L.block, L.blocks_per_sm, L.num_sms, s);
}

}  // namespace mci
