// box.cu -- history-based transport of the two-region multigroup box.
//
// A persistent kernel with lane refill (as for the slab) follows one
// particle per lane.  Work items are either source histories (a ticket over
// global history indices) or the split children waiting in a device bank.
// Children created by a launch are appended to the other bank; the host then
// launches the next generation on them, until a generation creates none.
// Every particle's stream depends only on its own seed (Eq. 3/4 for sources,
// Eq. 5 for children), so the generation order changes no result, and the
// int64 mesh tally is bit-identical to any other schedule.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "box.cuh"
#include "internal.h"
#include "transport.h"

namespace {

using mcb::BoxDev;
using mcb::ChildRec;

__global__ void box_prep_kernel(BoxDev* __restrict__ p, uint32_t n) {
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
    BoxDev& b = p[i];
    b.h = b.side / (double)b.mesh;
    b.inv_h = (double)b.mesh / b.side;
    mcx::fixed_of(b.inv_h, b.ih_q, b.ih_s);
    b.side_f = (float)b.side;
    b.lo_f = (float)b.lo;
    b.hi_f = (float)b.hi;
    b.h_f = b.side_f / (float)b.mesh;
    b.inv_h_f = (float)b.mesh / b.side_f;
    bool ok = b.side >= 0x1p-40 && b.side <= 0x1p40;
    for (int r = 0; r < 2; ++r) {
      ok = ok && b.ws[r] >= 0x1p-60 && b.ws[r] <= 0x1p60;
      b.inv_ws_f[r] = 1.0f / (float)b.ws[r];
      b.inv_st[r] = 1.0 / b.st[r];
      b.inv_st_f[r] = 1.0f / (float)b.st[r];
      b.c_f[r] = (float)b.c[r];
      b.wl_f[r] = (float)b.wl[r];
      b.wh_f[r] = (float)b.wh[r];
      b.ws_f[r] = (float)b.ws[r];
      for (int g = 0; g < mcb::kMaxG; ++g)
        for (int k = 0; k < mcb::kMaxG; ++k) b.cdf_n[r][g][k] = mcb::cdf_threshold(b.cdf[r][g][k]);
    }
    b.f32_ok = ok ? 1u : 0u;
    const uint64_t parent = b.seeding == MC_SEED_HASH_HIER ? mcd::hash64(b.key, b.seed) : b.seed;
    b.seed_hash = mcd::seed_hash_of(parent);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t acc = 0;
    for (uint32_t i = 0; i < n; ++i) {
      p[i].hist_begin = acc;
      acc += p[i].n_hist;
    }
  }
}

struct BoxArgs {
  const BoxDev* probs;
  uint32_t nprob;
  uint32_t chunk;
  const ChildRec* child_in;  // nullptr: the work items are source histories
  uint64_t range_begin, total;
  unsigned long long* ticket;
  ChildRec* child_out;
  unsigned long long* child_out_count;
  uint64_t child_cap;
  unsigned long long* tally;
  unsigned long long* counts;
  uint64_t* hist_state;
  uint64_t* hist_draws;
  mcd::Lcg lcg;
  uint64_t event_cap;
  mcd::Pow2Maps pow2;
};

__device__ __forceinline__ uint32_t find_box(const BoxDev* p, uint32_t n, uint64_t gi) {
  uint32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (p[mid].hist_begin <= gi) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Where a lane stands between two phases of the kernel's loop.
enum LaneState : int {
  kDead = 0,   // no particle
  kReady,      // next: a flight
  kWalking,    // its flight is being tallied
  kArrived,    // the tally of its flight is complete
  kInverse,    // a split child: its direction needs its inverse
  kSource,     // a source particle without a direction
  kCollided,   // at a collision site
  kEnded       // leaked, killed or capped: to be counted
};

// Lanes that wait before a warp refills, and pieces of its tally a lane
// makes per pass.  (Flat around these values: 3 to 8 lanes and 4 to 8 pieces
// are within 5 %; a pass makes 25.5 flights of 2.8 pieces each, at 12.7 lanes
// per piece, and refills every sixth time.)
template <typename T> constexpr int kRefillMin = sizeof(T) == 4 ? 3 : 4;
template <typename T> constexpr int kWalkSteps = sizeof(T) == 4 ? 5 : 4;
constexpr uint32_t kCountProbs = 16;  // problems whose counters a block keeps in shared memory

// fp32: bound by integer issue (80 % of the slots, at 15.7 lanes per
// instruction); fp64: by the fp64 unit (66 % busy at 17 lanes).  Each pass of
// the loop takes every live lane through the same phases -- refill, direction,
// flight, tally -- so that source and collision share one copy of the
// direction's code, a refill waits until some lanes need one, and a flight
// whose track crosses many voxels does not hold its warp.  Particle, walk and
// axis state are scalars, none of them indexed (fp32 spills some 80 bytes at
// its 64 registers; in fp64 the rare call of surface_exact takes a copy of the
// particle through a 96-byte frame); a particle's counts go to its block's
// counters in shared memory when it ends.  Four blocks per SM in fp32 (64
// registers: 16.3 ms for 10^7 histories, 17.4 with three, 17.7 with five; 31.7
// before the phases), three in fp64 (80: 13.0 ms for 3 * 10^6, 45.7 before; four
// were 1 % slower).
template <int M, typename T, bool AGG, bool ONE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 3) box_history_kernel(const BoxArgs a) {
  __shared__ mcd::Affine tab[64];
  // A single problem's record is read on every flight: keep it in shared memory.
  __shared__ __align__(16) unsigned char s_prob[ONE ? sizeof(BoxDev) : 16];
  // fp64, one problem: its mesh planes, read on every voxel crossing
  __shared__ double s_planes[ONE && sizeof(T) == 8 ? mcb::kMaxPlanes : 1];
  __shared__ unsigned long long s_counts[kCountProbs * MC_NCOUNT];
  mcd::load_maps(a.pow2, tab);
  const bool block_counts = ONE || a.nprob <= kCountProbs;
  if (block_counts)
    for (uint32_t i = threadIdx.x; i < a.nprob * MC_NCOUNT; i += blockDim.x) s_counts[i] = 0ull;
  if constexpr (ONE) {
    const uint64_t* src = reinterpret_cast<const uint64_t*>(a.probs);
    uint64_t* dst = reinterpret_cast<uint64_t*>(s_prob);
    for (uint32_t i = threadIdx.x; i < sizeof(BoxDev) / 8; i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
  const BoxDev* const probs = ONE ? reinterpret_cast<const BoxDev*>(s_prob) : a.probs;
  const double* const planes = ONE && sizeof(T) == 8 ? s_planes : nullptr;
  if constexpr (ONE && sizeof(T) == 8) {
    for (uint32_t j = threadIdx.x; j <= probs->mesh; j += blockDim.x) s_planes[j] = mcb::plane_of(*probs, (int)j);
    __syncthreads();
  }
  unsigned long long* const counts = block_counts ? s_counts : a.counts;
  const unsigned kFull = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned lt_mask = (1u << lane) - 1u;
  const mcd::Lcg l = a.lcg;

  uint64_t pool_next = 0, pool_end = 0;
  bool more = true, primary = false;
  int state = kDead, outcome = 0;
  const BoxDev* P = probs;  // (ONE: never changes, nor does pi)
  uint32_t pi = 0, ncoll = 0;
  mcs::Rng<M> r{0ull, 0ull};
  mcb::Part<T> q{};
  mcb::Walk<T> k{};
  uint64_t gi = 0, events = 0, tbase = 0;

  for (;;) {
    // New items once enough lanes wait for one: a refill (seed, source draws,
    // record loads) costs the warp the same for one lane as for many.
    unsigned dead = __ballot_sync(kFull, state == kDead);
    if (more && (__popc(dead) >= kRefillMin<T> || dead == kFull)) {
      while (dead != 0u && more) {
        if (pool_next >= pool_end) {
          unsigned long long b0 = 0;
          if (lane == 0) b0 = atomicAdd(a.ticket, (unsigned long long)a.chunk);
          b0 = __shfl_sync(kFull, b0, 0);
          if (b0 >= a.total) { more = false; break; }
          pool_next = b0;
          pool_end = min((uint64_t)b0 + (uint64_t)a.chunk, (uint64_t)a.total);
        }
        const uint64_t avail = pool_end - pool_next;
        const unsigned rank = __popc(dead & lt_mask);
        if (state == kDead && rank < avail) {
          const uint64_t item = pool_next + rank;
          if (a.child_in == nullptr) {
            gi = a.range_begin + item;
            if constexpr (!ONE) {
              pi = find_box(a.probs, a.nprob, gi);
              P = probs + pi;
            }
            const uint64_t id = gi - P->hist_begin;
            const uint64_t nvox = (uint64_t)P->mesh * P->mesh * P->mesh;
            tbase = P->tally_offset;
            if (P->n_batches > 1) tbase += mcs::batch_of(id, P->n_hist, P->n_batches) * nvox;
            const uint64_t seed = P->seeding == MC_SEED_STRIDE
                                      ? mcs::skip_tab(tab, P->seed, P->stride_q * (P->id_offset + id)) & l.mask
                                      : mcd::hash_with(id, P->seed_hash) & l.mask;
            r = mcs::Rng<M>{seed, 0ull};
            mcb::source_position<M, T>(*P, r, l, q);
            primary = true;
            atomicAdd(counts + (size_t)pi * MC_NCOUNT + MC_C_SOURCE, 1ull);
            state = kSource;
          } else {
            const ChildRec& c = a.child_in[item];
            if constexpr (!ONE) {
              pi = c.prob;
              P = probs + pi;
            }
            tbase = c.tbase;
            r = mcs::Rng<M>{c.rng, 0ull};
            mcb::child_state<T>(c, q);
            primary = false;
            state = kInverse;
          }
          mcb::walk_locate<T>(*P, q, k);
          events = 0;
          ncoll = 0;
        }
        pool_next += min((uint64_t)__popc(dead), avail);
        dead = __ballot_sync(kFull, state == kDead);
      }
      if (dead == kFull) break;  // no particle left, and no item
    } else if (dead == kFull) {
      break;
    }

    // Directions: of source particles and of collided ones on one code path.
    if (state >= kInverse) {
      if (state == kCollided) mcb::collide_group<M, T>(*P, r, l, q);
      if (state != kInverse) mcb::iso_dir<M, T>(r, l, q.u);
      mcb::set_inv(q);
      if (state == kCollided) {
        ++ncoll;
        outcome = mcb::weight_window<M, T>(*P, r, l, q);
        if (outcome >= mcb::kSplitBase) {
          const uint32_t n = (uint32_t)(outcome - mcb::kSplitBase);
          unsigned long long* c = counts + (size_t)pi * MC_NCOUNT;
          atomicAdd(c + MC_C_SPLITS, 1ull);
          atomicAdd(c + MC_C_CHILDREN, (unsigned long long)(n - 1));
          for (uint32_t i = 0; i + 1 < n; ++i) {
            const unsigned long long idx = atomicAdd(a.child_out_count, 1ull);
            if (idx < a.child_cap) {
              mcb::store_child<T>(a.child_out[idx], q, mcb::child_seed(i, r.x, l.mask), pi, tbase);
            }
          }
        }
      } else if (state == kSource) {
        q.region = mcb::region_of<T>(*P, q.p, q.u);
      }
      state = state == kCollided && outcome == mcb::kBoxKilled ? kEnded : kReady;
    }

    // Flights.
    if (state == kReady) {
      if (events == a.event_cap) {
        outcome = -1;
        state = kEnded;
      } else {
        ++events;
        T len;
        outcome = mcb::flight_length<M, T>(*P, r, l, q, len);
        mcb::walk_begin<T>(*P, q, len, planes, k);
        state = kWalking;
      }
    }

    // The tallies, at most kWalkSteps pieces per lane: the number of pieces
    // varies from lane to lane, and a lane with many goes on in the next
    // pass while the others take their next flight.
    for (int i = 0; i < kWalkSteps<T>; ++i) {
      if (__ballot_sync(kFull, state == kWalking) == 0u) break;
      if (state == kWalking && mcb::walk_step<T>(*P, q, k, a.tally + tbase, planes, AGG)) state = kArrived;
    }
    if (state == kArrived) {
      mcb::walk_leave<T>(*P, q, k);
      mcb::arrive<T>(q, k.L, outcome);
      state = outcome == mcb::kBoxCollide ? kCollided : (outcome == mcb::kBoxLeak ? kEnded : kReady);
    }

    if (state == kEnded) {
      unsigned long long* c = counts + (size_t)pi * MC_NCOUNT;
      atomicAdd(c + (outcome == mcb::kBoxLeak ? MC_C_LEAK_HI : outcome == mcb::kBoxKilled ? MC_C_ROULETTE_KILLS : MC_C_CAPPED),
                1ull);
      atomicAdd(c + MC_C_FLIGHTS, (unsigned long long)events);
      atomicAdd(c + MC_C_COLLISIONS, (unsigned long long)ncoll);
      atomicAdd(c + MC_C_SCATTERS, (unsigned long long)ncoll);
      atomicAdd(c + MC_C_DRAWS, (unsigned long long)r.draws);
      atomicMax(c + MC_C_MAX_DRAWS, (unsigned long long)r.draws);
      if (primary) {
        if (P->stride_q != 0 && r.draws > P->stride_q) {
          atomicAdd(c + MC_C_EXCEED_HIST, 1ull);
          atomicAdd(c + MC_C_EXCEED_DRAWS, (unsigned long long)(r.draws - P->stride_q));
        }
        if (a.hist_state) a.hist_state[gi] = r.x & l.mask;
        if (a.hist_draws) a.hist_draws[gi] = r.draws;
      }
      state = kDead;
    }
  }
  if (block_counts) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < a.nprob * MC_NCOUNT; i += blockDim.x) {
      const unsigned long long v = s_counts[i];
      if (v == 0ull) continue;
      if (i % MC_NCOUNT == MC_C_MAX_DRAWS) atomicMax(a.counts + i, v);
      else atomicAdd(a.counts + i, v);
    }
  }
}

}  // namespace

namespace {

// One problem, as most launches have (an instantiation of its own: the record
// and the planes at fixed places in shared memory), or several.
template <int M, typename T, bool AGG>
void (*box_kernel_for(bool one))(const BoxArgs) {
  if constexpr (M == 63 && !AGG) {
    if (one) return box_history_kernel<M, T, AGG, true>;
  }
  (void)one;
  return box_history_kernel<M, T, AGG, false>;
}

template <int M, typename T, bool AGG>
int launch_box_gen(const BoxArgs& a, int block, int bps, int num_sms, cudaStream_t s) {
  auto k = box_kernel_for<M, T, AGG>(a.nprob == 1);
  int per_sm = bps;
  if (per_sm <= 0) {
    int st = mci::cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, 0),
                              "cudaOccupancyMaxActiveBlocksPerMultiprocessor(box)");
    if (st != MC_OK) return st;
    if (per_sm < 1) per_sm = 1;
  }
  const uint64_t warps_needed = (a.total + a.chunk - 1) / a.chunk;
  const uint64_t blocks_needed = (warps_needed * 32 + block - 1) / block;
  const uint64_t full = (uint64_t)num_sms * (uint64_t)per_sm;
  const int grid = (int)std::max<uint64_t>(1, std::min(full, blocks_needed));
  k<<<grid, block, 0, s>>>(a);
  return mci::cuda_status(cudaGetLastError(), "box_history_kernel launch");
}

template <int M, typename T>
int run_box_history(const mci::BoxLaunch& L, cudaStream_t s) {
  BoxArgs a{};
  a.probs = static_cast<const BoxDev*>(L.d_probs);
  a.nprob = L.n_problems;
  a.chunk = L.chunk;
  a.tally = reinterpret_cast<unsigned long long*>(L.tally->d_bins);
  a.counts = reinterpret_cast<unsigned long long*>(L.tally->d_counts);
  a.hist_state = L.tally->d_hist_state;
  a.hist_draws = L.tally->d_hist_draws;
  a.lcg = mcd::Lcg{L.lcg.g, L.lcg.c, mcd::mask_of(L.lcg.m), L.lcg.m};
  a.event_cap = L.event_cap;
  a.pow2 = mcd::pow2_maps(L.lcg.g, L.lcg.c);
  a.ticket = L.d_ticket;
  a.child_cap = L.child_cap;
  ChildRec* bank[2] = {static_cast<ChildRec*>(L.d_child[0]), static_cast<ChildRec*>(L.d_child[1])};
  unsigned long long* cnt[2] = {L.d_child_count, L.d_child_count + 1};
  for (uint64_t start = 0; start < L.total; start += L.primary_chunk) {
    const uint64_t n = std::min<uint64_t>(L.primary_chunk, L.total - start);
    // generation 0: source histories
    MC_TRY_CUDA(cudaMemsetAsync(L.d_ticket, 0, sizeof(unsigned long long), s));
    MC_TRY_CUDA(cudaMemsetAsync(cnt[0], 0, sizeof(unsigned long long), s));
    a.child_in = nullptr;
    a.range_begin = L.range_begin + start;
    a.total = n;
    a.child_out = bank[0];
    a.child_out_count = cnt[0];
    int st = (L.tally_agg ? launch_box_gen<M, T, true> : launch_box_gen<M, T, false>)(a, L.block, L.blocks_per_sm, L.num_sms, s);
    if (st != MC_OK) return st;
    int cur = 0;
    for (int gen = 1;; ++gen) {
      unsigned long long made = 0;
      MC_TRY_CUDA(cudaMemcpyAsync(L.h_count, cnt[cur], sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
      MC_TRY_CUDA(cudaStreamSynchronize(s));
      made = *L.h_count;
      if (made > L.child_cap) {
        mci::set_error("box transport: %llu children in one generation exceed the bank of %llu", made,
                       (unsigned long long)L.child_cap);
        return MC_ERR_CAPACITY;
      }
      if (made == 0) break;
      if ((uint32_t)gen > L.max_generations) {
        mci::set_error("box transport: more than %u generations of children", L.max_generations);
        return MC_ERR_TIMEOUT;
      }
      const int nxt = cur ^ 1;
      MC_TRY_CUDA(cudaMemsetAsync(L.d_ticket, 0, sizeof(unsigned long long), s));
      MC_TRY_CUDA(cudaMemsetAsync(cnt[nxt], 0, sizeof(unsigned long long), s));
      a.child_in = bank[cur];
      a.range_begin = 0;
      a.total = made;
      a.child_out = bank[nxt];
      a.child_out_count = cnt[nxt];
      st = (L.tally_agg ? launch_box_gen<M, T, true> : launch_box_gen<M, T, false>)(a, L.block, L.blocks_per_sm, L.num_sms, s);
      if (st != MC_OK) return st;
      cur = nxt;
    }
  }
  return MC_OK;
}

}  // namespace

namespace mci {

size_t box_dev_size() { return sizeof(BoxDev); }
size_t box_child_rec_size() { return sizeof(ChildRec); }

int box_fill_host(const mc_problem* src, uint32_t n, void* dst) {
  BoxDev* d = static_cast<BoxDev*>(dst);
  for (uint32_t i = 0; i < n; ++i) {
    const mc_box_spec* b = src[i].box;
    BoxDev q;
    std::memset(&q, 0, sizeof q);
    q.side = b->side;
    q.lo = b->inner_lo;
    q.hi = b->inner_hi;
    for (int r = 0; r < 2; ++r) {
      q.st[r] = b->sigma_t[r];
      q.c[r] = b->c[r];
      q.wl[r] = b->ww_low[r];
      q.wh[r] = b->ww_high[r];
      q.ws[r] = b->ww_survive[r];
      for (int g = 0; g < MC_BOX_MAX_GROUPS; ++g)
        for (int h = 0; h < MC_BOX_MAX_GROUPS; ++h) q.cdf[r][g][h] = b->scatter_cdf[r][g][h];
    }
    q.ng = b->n_groups;
    q.mesh = b->mesh;
    q.max_split = b->max_split;
    q.n_hist = src[i].n_histories;
    q.seed = src[i].seed;
    q.stride_q = src[i].stride_q;
    q.id_offset = src[i].id_offset;
    q.key = src[i].key;
    q.tally_offset = src[i].tally_offset;
    q.n_batches = src[i].n_batches;
    q.seeding = src[i].seeding;
    q.source = src[i].source;
    d[i] = q;
  }
  return MC_OK;
}

int box_prep(void* d_probs, uint32_t n, cudaStream_t s) {
  box_prep_kernel<<<1, 256, 0, s>>>(static_cast<BoxDev*>(d_probs), n);
  return cuda_status(cudaGetLastError(), "box_prep_kernel launch");
}

int box_history_run(const BoxLaunch& L, cudaStream_t s) {
  if (L.lcg.m == 63) return L.f32 ? run_box_history<63, float>(L, s) : run_box_history<63, double>(L, s);
  return L.f32 ? run_box_history<0, float>(L, s) : run_box_history<0, double>(L, s);
}

}  // namespace mci
