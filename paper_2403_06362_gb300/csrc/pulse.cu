// pulse.cu -- the supercritical, time-dependent pulse problem of Section 5:
// a pulse at t = x = 0 in an infinite homogeneous medium, scattering with
// multiplicity (k = c * nu > 1), census at t_end, and the collision-estimator
// flux averaged over [-x_half, x_half] in unit time bins, tallied per
// (repetition, batch).
//
// History-based: a lane follows one source particle and its family of
// secondaries depth-first.  Those that wait are records on the lane's stack in
// device memory.  In hash mode each secondary owns a stream seeded on demand by
// S_c = hash(k, S_p) (Section 4, Eq. 5), so a record holds all secondaries of a
// collision, the newest record stays in registers, and when the sources have run
// out, lanes with nothing left take the oldest record of a lane of their warp:
// who follows a secondary changes no result.  In stride mode the family shares
// the source particle's stream, which fixes the depth-first order the
// secondaries are drawn in -- the sequential bookkeeping the paper's hashing
// removes -- and its records hold one each and stay with their lane.
// The fp64 arithmetic is rounded once per operation (--fmad=false).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "internal.h"
#include "mc_log.cuh"
#include "pulse.cuh"
#include "slab.cuh"
#include "transport.h"

namespace {

using mcp::Overflow;
using mcp::PulseDev;
using mcp::pulse_seed;

struct PulseArgs {
  const PulseDev* prob;
  uint64_t range_begin, total;
  uint32_t chunk;
  unsigned long long* ticket;
  unsigned long long* tally;
  unsigned long long* counts;
  uint64_t* hist_state;
  uint64_t* hist_draws;
  mcd::Lcg lcg;
  uint64_t event_cap;
  uint32_t stack_depth;            // pending secondaries a lane keeps (<= kStack)
  mcp::StackRec* stack;            // [stack_depth][threads of the launch]
  const Overflow* ovf_in;          // non-null: the work items are overflowed secondaries
  const unsigned long long* ovf_in_count;
  Overflow* ovf_out;               // non-null (hash modes): where secondaries beyond the stack go
  unsigned long long* ovf_out_count;
  uint64_t ovf_cap;
  mcd::Pow2Maps pow2;              // stride
};

__global__ void pulse_prep_kernel(PulseDev* p) {
  if (threadIdx.x == 0) {
    p->inv_st = 1.0 / p->sigma_t;
    p->unit = __double2ll_rn(p->inv_st * mcs::kFix);
    p->seed_hash = mcd::seed_hash_of(p->seed);
    p->c_n = (uint64_t)ceil(p->c * 0x1p53);
    // floor(nu + u) over u = n 2^-53, n < 2^53, is floor(nu) or floor(nu) + 1
    // (nu <= 64) and does not decrease with n: the first n giving the larger
    // value, found with the same fp64 sum the transport definition uses
    const double fl = floor(p->nu);
    uint64_t lo = 0, hi = 1ull << 53;
    while (lo < hi) {
      const uint64_t mid = lo + ((hi - lo) >> 1);
      if (floor(p->nu + (double)mid * 0x1p-53) > fl) hi = mid;
      else lo = mid + 1;
    }
    p->nu_n = lo;
    p->nu_floor = (uint32_t)fl;
  }
}

// A lane's counts, few enough to stay in registers beside the particle.
// Collisions, absorptions and the rest follow from them: a flight ends at the
// census or collides, a collision scatters or absorbs.  Event caps, dropped
// secondaries and exceedances go to the block's counters in shared memory.
// N: on 32 bits they are flushed now and then; 64 bits never need it.
template <typename N>
struct PulseCounts {
  N src, flights, census, scat, children;
  uint64_t draws, maxd;
  __device__ void flush(unsigned long long* c) {
    if (src) atomicAdd(c + MC_C_SOURCE, (unsigned long long)src);
    if (flights) atomicAdd(c + MC_C_FLIGHTS, (unsigned long long)flights);
    const N coll = flights - census;
    if (coll) atomicAdd(c + MC_C_COLLISIONS, (unsigned long long)coll);
    if (coll != scat) atomicAdd(c + MC_C_ABSORPTIONS, (unsigned long long)(coll - scat));
    if (scat) atomicAdd(c + MC_C_SCATTERS, (unsigned long long)scat);
    if (census) atomicAdd(c + MC_C_LEAK_HI, (unsigned long long)census);
    if (children) atomicAdd(c + MC_C_CHILDREN, (unsigned long long)children);
    if (draws) atomicAdd(c + MC_C_DRAWS, (unsigned long long)draws);
    if (maxd) atomicMax(c + MC_C_MAX_DRAWS, (unsigned long long)maxd);
    src = flights = census = scat = children = 0;
    draws = maxd = 0ull;
  }
};

// Lanes that wait for a source before a warp refills (its seeds, three
// hashes each, cost the warp the same for one lane as for many), and, once
// the sources have run out, before it hands pending secondaries to them.
constexpr int kRefillMin = 3;
constexpr int kShareMin = 8;

// Bound by integer issue (the logarithm; 3 * 10^6 sources: 68 % of the slots at
// 20 lanes per instruction).  A lane follows a source particle and its family
// depth first.  Hash seeds: the secondaries of a collision are one record,
// the newest of which stays in registers (their seeds are hashed one by one
// as they are taken), so most collisions touch no memory; and when the
// sources have run out, lanes with nothing left take records from the lanes
// of their warp that still hold some -- a stream depends on its seed alone,
// so who follows it changes nothing.  (Stride: the family shares one stream
// in depth-first order, so its secondaries stay with their lane.)  Against
// one record per secondary, all in memory, and no sharing: 58.0 -> 40.4 ms for
// 3 * 10^7 sources (29.7 -> 16.7 warp instructions per flight at 12.2 -> 20.7
// lanes; 52.0 ms without the sharing), 3.4 -> 0.5 ms for 5000; 37.9 ms with
// 2u - 1 by a subtraction.  Hash at 64 registers (at 84 a seventh slower).
// Stride runs wait for a family's one chain of events until many lanes carry
// one: a scattered particle draws its direction in place, and the row's place
// is kept with 64-bit counts that need no flush (5000 sources 4.32 -> 3.86 ms,
// 6 * 10^6 13.8 -> 13.0 at 80 registers; 4.09 and 13.4 held at 72).
template <int M, bool HASH, bool AGG>
__global__ void __launch_bounds__(256, HASH ? 4 : 1) pulse_kernel(const PulseArgs a) {
  __shared__ mcd::Affine tab[64];
  __shared__ PulseDev sP;
  __shared__ unsigned long long s_counts[MC_NCOUNT];
  if constexpr (!HASH) mcd::load_maps(a.pow2, tab);
  if (threadIdx.x == 0) sP = *a.prob;
  for (uint32_t i = threadIdx.x; i < MC_NCOUNT; i += blockDim.x) s_counts[i] = 0ull;
  __syncthreads();
  const PulseDev& P = sP;
  const mcd::Lcg l = a.lcg;
  const unsigned kFull = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;

  const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
  mcp::StackRec* const my_stack = a.stack + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  // the lane's records in memory: sp of them, from the lo-th of its
  // stack_depth entries on, round the end (at most pend - left, so they fit)
  uint32_t lo = 0, sp = 0;
  auto entry = [&](uint32_t k) {
    if constexpr (!HASH) return my_stack + (uint64_t)k * nthreads;  // lo stays 0
    const uint32_t i = lo + k;
    return my_stack + (uint64_t)(i >= a.stack_depth ? i - a.stack_depth : i) * nthreads;
  };
  // hash: the newest record, in registers; `left` secondaries of it are not
  // yet taken, `pend` wait in all
  double tx = 0.0, tt = 0.0;
  uint64_t ts = 0;
  uint32_t left = 0, pend = 0;
  uint64_t pool_next = 0, pool_end = 0;
  bool more = true, alive = false, primary = false;
  PulseCounts<std::conditional_t<HASH, uint32_t, uint64_t>> lc{};
  mcs::Rng<M> r{0ull, 0ull};
  double x = 0.0, t = 0.0, mu = 0.0;
  uint64_t gi = 0, events = 0;
  uint32_t grp = 0;
  unsigned long long* row = nullptr;  // stride: the family's tally row
  const uint64_t total = a.ovf_in ? min((uint64_t)*a.ovf_in_count, a.ovf_cap) : a.total;

  for (;;) {
    unsigned dead = __ballot_sync(kFull, !alive);
    if (more && (__popc(dead) >= kRefillMin || dead == kFull)) {
      while (dead != 0u && more) {
        if (pool_next >= pool_end) {
          unsigned long long b0 = 0;
          if (lane == 0) b0 = atomicAdd(a.ticket, (unsigned long long)a.chunk);
          b0 = __shfl_sync(kFull, b0, 0);
          if (b0 >= total) { more = false; break; }
          pool_next = b0;
          pool_end = min((uint64_t)b0 + (uint64_t)a.chunk, total);
        }
        const uint64_t avail = pool_end - pool_next;
        const unsigned rank = __popc(dead & lt_mask);
        if (!alive && rank < avail) {
          if (a.ovf_in) {
            // an overflowed secondary: hash seeded, it starts a family of its own
            const Overflow e = a.ovf_in[pool_next + rank];
            grp = e.group;
            r = mcs::Rng<M>{e.seed, 0ull};
            x = e.x;
            t = e.t;
            primary = false;
          } else {
            gi = a.range_begin + pool_next + rank;
            grp = mcp::pulse_group(P, gi);
            r = mcs::Rng<M>{pulse_seed(P, gi, grp, tab, l.mask), 0ull};
            x = 0.0;
            t = 0.0;
            primary = true;
            ++lc.src;
          }
          mu = mcx::two_u_minus_1(r.next_n(l));
          if constexpr (!HASH) row = a.tally + P.tally_offset + (uint64_t)grp * P.n_time_bins;
          events = 0;
          alive = true;
        }
        pool_next += min((uint64_t)__popc(dead), avail);
        dead = __ballot_sync(kFull, !alive);
      }
    }
    if (dead == kFull) break;  // (while there are sources, the refill leaves some lane alive)
    bool take = false;  // the lane's next particle is the newest record's next secondary
    if constexpr (HASH) {
      if (!more && __popc(dead) >= kShareMin) {
        // the r-th lane without a particle takes a record of the r-th lane that has one to spare
        const unsigned donors = __ballot_sync(kFull, alive && pend != 0u);
        if (donors != 0u) {
          const unsigned rank = __popc((alive ? donors : dead) & lt_mask);
          const bool give = alive && pend != 0u && rank < (unsigned)__popc(dead);
          double rx = tx, rt = tt;
          uint64_t rs = ts;
          uint32_t rl = left;
          if (give) {
            if (sp != 0u) {  // its oldest
              mcp::stack_get(entry(0u), rx, rt, rs, rl);
              --sp;
              lo = lo + 1u == a.stack_depth ? 0u : lo + 1u;
            } else {
              left = 0u;
            }
            pend -= rl;
          }
          const bool get = !alive && rank < (unsigned)__popc(donors);
          unsigned m = donors;
          for (unsigned i = 0; get && i < rank; ++i) m &= m - 1u;
          const int from = get ? __ffs((int)m) - 1 : (int)lane;
          rx = __shfl_sync(kFull, rx, from);
          rt = __shfl_sync(kFull, rt, from);
          rs = __shfl_sync(kFull, rs, from);
          rl = __shfl_sync(kFull, rl, from);
          const uint32_t rg = __shfl_sync(kFull, grp, from);
          if (get) {
            tx = rx;
            tt = rt;
            ts = rs;
            left = pend = rl;
            grp = rg;
            take = alive = true;
            primary = false;
          }
        }
      }
    }

    bool redraw = take;
    if (alive && !take) {
      bool ended = false;
      if (events == a.event_cap) {
        atomicAdd(s_counts + MC_C_CAPPED, 1ull);
        ended = true;
      } else {
        ++events;
        ++lc.flights;
        const double d = mclog::neglog1m_n(r.next_n(l)) * P.inv_st;
        const double tn = t + d;
        if (!mcs::nn_lt(tn, P.t_end)) {  // tn >= t_end, both non-negative
          ++lc.census;
          ended = true;
        } else {
          const double xn = x + d * mu;
          if (mcx::abs_le(xn, P.x_half)) {
            // (t_end is at most 10^6.  The short form: stride 14.5 -> 14.3 ms; hash at
            // its 64 registers 37.9 -> 39.1 ms)
            const uint64_t jf = HASH ? mcx::floor_nonneg(tn) : mcx::floor_small(tn);
            const uint32_t j = jf < P.n_time_bins ? (uint32_t)jf : P.n_time_bins - 1;
            unsigned long long* const slot =
                HASH ? a.tally + P.tally_offset + (uint64_t)grp * P.n_time_bins + j : row + j;
            if constexpr (AGG) mcd::warp_agg_add(slot, (unsigned long long)P.unit);
            else atomicAdd(slot, (unsigned long long)P.unit);
          }
          x = xn;
          t = tn;
          if (r.next_n(l) < P.c_n) {  // u < c
            ++lc.scat;
            const uint32_t n = P.nu_floor + (r.next_n(l) >= P.nu_n ? 1u : 0u);  // floor(nu + u)
            if constexpr (HASH) {
              const uint32_t kids = n - 1u, room = a.stack_depth - pend, fit = min(kids, room);
              if (fit != 0u) {
                if (left != 0u) {
                  mcp::stack_put(entry(sp), tx, tt, ts, left);
                  ++sp;
                }
                tx = x;
                tt = t;
                ts = r.x & l.mask;
                left = fit;
                pend += fit;
              }
              for (uint32_t k = fit; k < kids; ++k) {  // a full stack: to the overflow bank
                const unsigned long long idx = atomicAdd(a.ovf_out_count, 1ull);
                if (idx < a.ovf_cap) a.ovf_out[idx] = Overflow{x, t, mcd::hash64(k, r.x & l.mask) & l.mask, grp, 0u};
                else atomicAdd(s_counts + MC_C_DROPPED, 1ull);  // reported as MC_ERR_CAPACITY by mc_tally_read
                lc.children += idx < a.ovf_cap ? 1u : 0u;
              }
              lc.children += fit;
            } else {
              for (uint32_t k = 0; k + 1 < n; ++k) {
                if (sp < a.stack_depth) {
                  mcp::stack_put(entry(sp), x, t, 0ull, 1u);
                  ++sp;
                  ++lc.children;
                } else {
                  atomicAdd(s_counts + MC_C_DROPPED, 1ull);
                }
              }
            }
            // its new direction: below, on the code path a new particle shares
            // (hash), or here, one branch sooner (stride)
            if constexpr (HASH) redraw = true;
            else mu = mcx::two_u_minus_1(r.next_n(l));
          } else {
            ended = true;
          }
        }
      }
      if (ended) {  // the current particle ended
        if (HASH || sp == 0u) {  // and with it its stream
          lc.draws += r.draws;
          if (r.draws > lc.maxd) lc.maxd = r.draws;
          if (!HASH || primary) {
            if (a.hist_state) a.hist_state[gi] = r.x & l.mask;
            if (a.hist_draws) a.hist_draws[gi] = r.draws;
            if (P.stride_q != 0 && r.draws > P.stride_q) {
              atomicAdd(s_counts + MC_C_EXCEED_HIST, 1ull);
              atomicAdd(s_counts + MC_C_EXCEED_DRAWS, (unsigned long long)(r.draws - P.stride_q));
            }
          }
        }
        primary = false;
        events = 0;
        if constexpr (HASH) {
          take = pend != 0u;
          alive = take;
        } else {
          alive = sp != 0u;
          if (alive) {  // the next secondary of the family, on the family's stream
            --sp;
            uint64_t s;
            uint32_t n;
            mcp::stack_get(entry(sp), x, t, s, n);
          }
        }
        redraw = alive;
        if (HASH && lc.flights > (1u << 24)) lc.flush(a.counts);  // (up to 63 secondaries each)
      }
    }
    if constexpr (HASH) {
      if (take) {  // Eq. (5)
        --pend;
        --left;
        x = tx;
        t = tt;
        r = mcs::Rng<M>{mcd::hash64((uint64_t)left, ts) & l.mask, 0ull};
        events = 0;
        if (left == 0u && sp != 0u) {
          --sp;
          mcp::stack_get(entry(sp), tx, tt, ts, left);
        }
      }
    }
    // the direction of a new particle and (hash) of a scattered one
    if (redraw) mu = mcx::two_u_minus_1(r.next_n(l));
  }
  // the lanes' counts, summed over the warp (they share a cache line)
  {
    const unsigned long long so = mcd::warp_sum64(lc.src), fl = mcd::warp_sum64(lc.flights),
                             ce = mcd::warp_sum64(lc.census), sc = mcd::warp_sum64(lc.scat),
                             ch = mcd::warp_sum64(lc.children), dr = mcd::warp_sum64(lc.draws),
                             mx = mcd::warp_max64(lc.maxd);
    if (lane == 0) {
      atomicAdd(s_counts + MC_C_SOURCE, so);
      atomicAdd(s_counts + MC_C_FLIGHTS, fl);
      atomicAdd(s_counts + MC_C_COLLISIONS, fl - ce);
      atomicAdd(s_counts + MC_C_ABSORPTIONS, fl - ce - sc);
      atomicAdd(s_counts + MC_C_SCATTERS, sc);
      atomicAdd(s_counts + MC_C_LEAK_HI, ce);
      atomicAdd(s_counts + MC_C_CHILDREN, ch);
      atomicAdd(s_counts + MC_C_DRAWS, dr);
      atomicMax(s_counts + MC_C_MAX_DRAWS, mx);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < MC_NCOUNT; i += blockDim.x) {
    const unsigned long long v = s_counts[i];
    if (v == 0ull) continue;
    if (i == MC_C_MAX_DRAWS) atomicMax(a.counts + i, v);
    else atomicAdd(a.counts + i, v);
  }
}

}  // namespace

namespace mci {

size_t pulse_dev_size() { return sizeof(PulseDev); }

int pulse_fill_host(const mc_problem* src, void* dst) {
  PulseDev q;
  std::memset(&q, 0, sizeof q);
  const mc_pulse_spec* s = src->pulse;
  q.c = s->c;
  q.nu = s->nu;
  q.t_end = s->t_end;
  q.x_half = s->x_half;
  q.sigma_t = s->sigma_t;
  q.n_hist = src->n_histories;
  q.seed = src->seed;
  q.stride_q = src->stride_q;
  q.id_offset = src->id_offset;
  q.tally_offset = src->tally_offset;
  q.n_reps = s->n_reps;
  q.n_batches = s->n_batches;
  q.per_batch = s->per_batch;
  q.n_time_bins = s->n_time_bins;
  q.seeding = src->seeding;
  q.n_census = s->n_census;
  q.pc_target = s->pc_target;
  std::memcpy(dst, &q, sizeof q);
  return MC_OK;
}

int pulse_prep(void* d_prob, cudaStream_t s) {
  pulse_prep_kernel<<<1, 32, 0, s>>>(static_cast<PulseDev*>(d_prob));
  return cuda_status(cudaGetLastError(), "pulse_prep_kernel launch");
}

// The kernel variant for the LCG width, the seeding mode and the tally atomics.
static void (*pulse_kernel_for(uint32_t m, bool hash, bool agg))(const PulseArgs) {
  if (agg) return m == 63 ? (hash ? pulse_kernel<63, true, true> : pulse_kernel<63, false, true>)
                          : (hash ? pulse_kernel<0, true, true> : pulse_kernel<0, false, true>);
  return m == 63 ? (hash ? pulse_kernel<63, true, false> : pulse_kernel<63, false, false>)
                 : (hash ? pulse_kernel<0, true, false> : pulse_kernel<0, false, false>);
}

// The largest grid pulse_run launches for L (one persistent block per slot).
static int pulse_full_grid(const PulseLaunch& L, uint64_t* full_out) {
  const bool hash = L.seeding != MC_SEED_STRIDE;
  auto k = pulse_kernel_for(L.lcg.m, hash, L.tally_agg);
  int per_sm = 0;
  int st = cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, L.block, 0),
                       "cudaOccupancyMaxActiveBlocksPerMultiprocessor(pulse)");
  if (st != MC_OK) return st;
  if (per_sm < 1) per_sm = 1;
  *full_out = (uint64_t)L.num_sms * per_sm;
  return MC_OK;
}

int pulse_stack_bytes(const PulseLaunch& L, size_t* bytes) {
  uint64_t full = 0;
  const int st = pulse_full_grid(L, &full);
  if (st != MC_OK) return st;
  *bytes = (size_t)full * (size_t)L.block * L.stack_depth * sizeof(mcp::StackRec);
  return MC_OK;
}

int pulse_run(const PulseLaunch& L, cudaStream_t s) {
  PulseArgs a{};
  a.prob = static_cast<const PulseDev*>(L.d_prob);
  a.range_begin = L.range_begin;
  a.total = L.total;
  a.chunk = L.chunk;
  a.ticket = L.d_ticket;
  a.tally = reinterpret_cast<unsigned long long*>(L.tally->d_bins);
  a.counts = reinterpret_cast<unsigned long long*>(L.tally->d_counts);
  a.hist_state = L.tally->d_hist_state;
  a.hist_draws = L.tally->d_hist_draws;
  a.lcg = mcd::Lcg{L.lcg.g, L.lcg.c, mcd::mask_of(L.lcg.m), L.lcg.m};
  a.event_cap = L.event_cap;
  a.pow2 = mcd::pow2_maps(L.lcg.g, L.lcg.c);
  a.stack_depth = L.stack_depth;
  a.stack = static_cast<mcp::StackRec*>(L.d_stack);
  const bool hash = L.seeding != MC_SEED_STRIDE;
  auto k = pulse_kernel_for(L.lcg.m, hash, L.tally_agg);
  uint64_t full = 0;
  int st = pulse_full_grid(L, &full);
  if (st != MC_OK) return st;
  if (!L.d_stack || L.stack_bytes < (size_t)full * L.block * L.stack_depth * sizeof(mcp::StackRec)) {
    set_error("pulse transport: the lane stacks need more device memory than was given");
    return MC_ERR_ARG;
  }
  const uint64_t warps_needed = (a.total + a.chunk - 1) / a.chunk;
  const uint64_t blocks_needed = (warps_needed * 32 + L.block - 1) / L.block;
  const int grid = (int)std::max<uint64_t>(1, std::min<uint64_t>(full, blocks_needed));
  if (!L.d_ovf) {
    k<<<grid, L.block, 0, s>>>(a);
    return cuda_status(cudaGetLastError(), "pulse_kernel launch");
  }
  // Hash modes: secondaries beyond the lane stacks go to an overflow bank,
  // processed generation by generation until a generation overflows nothing.
  auto* cnt = static_cast<unsigned long long*>(L.d_ovf);
  Overflow* bank[2] = {reinterpret_cast<Overflow*>(static_cast<char*>(L.d_ovf) + 256),
                       reinterpret_cast<Overflow*>(static_cast<char*>(L.d_ovf) + 256 + L.ovf_cap * sizeof(Overflow))};
  a.ovf_cap = L.ovf_cap;
  a.ovf_out = bank[0];
  a.ovf_out_count = cnt;
  MC_TRY_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), s));
  k<<<grid, L.block, 0, s>>>(a);
  st = cuda_status(cudaGetLastError(), "pulse_kernel launch");
  for (int gen = 1; st == MC_OK; ++gen) {
    const int cur = (gen - 1) & 1, nxt = cur ^ 1;
    MC_TRY_CUDA(cudaMemcpyAsync(L.h_count, cnt + cur, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    MC_TRY_CUDA(cudaStreamSynchronize(s));
    const uint64_t made = std::min<uint64_t>(*L.h_count, L.ovf_cap);
    if (made == 0) break;
    if ((uint32_t)gen > L.max_generations) {
      set_error("pulse transport: more than %u generations of overflowed secondaries", L.max_generations);
      return MC_ERR_TIMEOUT;
    }
    PulseArgs b = a;
    b.ovf_in = bank[cur];
    b.ovf_in_count = cnt + cur;
    b.ovf_out = bank[nxt];
    b.ovf_out_count = cnt + nxt;
    b.total = made;
    MC_TRY_CUDA(cudaMemsetAsync(cnt + nxt, 0, sizeof(unsigned long long), s));
    MC_TRY_CUDA(cudaMemsetAsync(L.d_ticket, 0, sizeof(unsigned long long), s));
    const uint64_t w = (made + a.chunk - 1) / a.chunk;
    const int g2 = (int)std::max<uint64_t>(1, std::min<uint64_t>(full, (w * 32 + L.block - 1) / L.block));
    k<<<g2, L.block, 0, s>>>(b);
    st = cuda_status(cudaGetLastError(), "pulse_kernel launch (overflow)");
  }
  return st;
}

size_t pulse_ovf_bytes(uint64_t cap) { return 256 + 2 * cap * sizeof(Overflow); }

}  // namespace mci
