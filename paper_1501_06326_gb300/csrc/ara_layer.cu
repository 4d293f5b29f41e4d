// The layer kernels of the ARA engine (Algorithm 1 with the secondary
// uncertainty of Section 3.3, per trial): k_gather streams the YET and finds
// the events of the layer's ELTs, k_losses draws the uniforms, inverts the
// Beta CDFs through the quantile tables, applies the ELT, occurrence and
// aggregate terms and writes the year losses.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "ara_internal.h"
#include "ara_window.cuh"

namespace ara {

// =============================================================== layer kernels
//
// k_gather: one persistent CTA of 32 warps per SM.  The CTA folds the layer's
// catalogue bitmap into a shared-memory membership filter once (as many words
// as shared memory holds; word w of the catalogue lands on w mod filt_words);
// then each warp independently takes tiles of kWarpTrials consecutive trials
// and streams the tile's YET ids, 256 per step (32 bytes per lane, not
// L1-allocated, two more steps in flight).  Each id is tested against the
// filter; the positives collect in a small ring, in YET order, and every 32 of
// them are resolved together against the rank directory (8 bytes: the word's
// bits and its pair base), a group's directory words in flight while the next
// step is filtered.  A member becomes an event record written in YET order to
// the tile's region of the event buffer.
// What bounds it is the SM's shared-memory and L1 data pipe (paper-1m: 79% of
// its wavefronts; about 80 a step, of which the filter's lookups with their
// bank conflicts take 27, the directory words 22, the id stream 16).  So the
// ring takes one packed word a positive, the lanes' places come from ballots
// and not from shuffles (which use that pipe too), groups are always full, and
// a trial is searched only where a group crosses into the next one: 99
// wavefronts a step before that and 311 warp instructions against 252; at
// paper-1m 1.37 ms before, 1.14 ms now.
//
// k_losses: each warp takes tiles and reads their records one per lane.  An
// event with one (event, ELT) pair is finished by its lane: Philox uniform,
// inverse Beta through the record's quantile table, ELT and occurrence terms,
// and a double-float add into the lane's sum for the event's trial.  Events
// with several pairs are queued and processed in windows of 32 pairs with a
// segmented sum; layers of many pairs an event take all events so.  Events
// with a pair whose record's table is not exact are deferred and resolved, 32
// at a time, by the FP32 Halley iteration.  At the end of a tile a
// reduce-scatter over the lanes gives the trials' sums, and the aggregate terms
// turn each into the trial's year loss.

namespace {

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

// Filter positives waiting to be resolved, per warp: up to 31 left from earlier
// steps and the 256 of one step.  kPacked: one word each, the event id above
// the low kPosBits bits of its position in the tile; else the id and the
// position in the step.
constexpr int kGatherRing = 288;
constexpr uint32_t kPosBits = 11;
constexpr int32_t kPackedCatalogue = 1 << (32 - kPosBits);

struct GatherWarp {
  int32_t off[16];            // trial offsets in the tile's positions; INT32_MAX past the tile's end
  uint32_t ring[kGatherRing];
};
struct GatherWarpWide {
  int32_t off[16];
  uint32_t ring[kGatherRing];
  uint8_t ring_q[kGatherRing];
};

template <bool kPacked>
using GatherShared = typename std::conditional<kPacked, GatherWarp, GatherWarpWide>::type;

}  // namespace

size_t gather_smem_bytes(int filt_words, int32_t catalogue) {
  return sizeof(uint32_t) * static_cast<size_t>(filt_words) +
         (catalogue <= kPackedCatalogue ? sizeof(GatherWarp) : sizeof(GatherWarpWide)) * (kGatherThreads / 32) + 16;
}

// k_gather's shared memory stays within the 196 KB carveout (less the 1 KB
// the driver reserves per block): the L1 that the rest of the SM's 256 KB
// leaves (60 KB) holds the id stream's loads in flight, and a larger carveout
// (L1 28 KB) was measured to slow the stream by a quarter, more than a larger
// filter saves.
constexpr int kGatherSmemBudget = 196 * 1024 - 1024;

int gather_filter_words(int64_t n_words, int max_smem, int32_t catalogue) {
  const int64_t budget = max_smem < kGatherSmemBudget ? max_smem : kGatherSmemBudget;
  const int64_t room = (budget - static_cast<int64_t>(gather_smem_bytes(0, catalogue))) / 4;
  const int64_t fw_max = room & ~int64_t(31);
  if (fw_max < 32) return 0;
  if (n_words <= 2 * fw_max) return static_cast<int>(n_words <= fw_max ? (n_words > 0 ? n_words : 1) : fw_max);
  int64_t fw = 32;
  while (fw * 2 <= fw_max) fw *= 2;
  return static_cast<int>(fw);
}

namespace {

// Eight YET ids (32 bytes, read once): not allocated in L1, whose capacity
// holds the loads in flight (measured 1% faster than evict-first loads).
struct Ids8 {
  uint32_t e[8];
};
__device__ __forceinline__ Ids8 ld_ids(const int32_t* a) {
  Ids8 v;
  asm("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v.e[0]), "=r"(v.e[1]), "=r"(v.e[2]), "=r"(v.e[3]), "=r"(v.e[4]), "=r"(v.e[5]), "=r"(v.e[6]), "=r"(v.e[7])
      : "l"(a));
  return v;
}

// State of one warp's pass over one tile.  Positions count from the 32-byte
// boundary at or below the tile's first event.
struct GatherTile {
  const int32_t* ids;  // position 0
  int32_t lead;        // positions before the tile's first event
  int32_t span;        // positions up to the tile's end
  uint2* out;          // the tile's region of the event buffer
  uint32_t nout;       // records written
  // the trial of the last position resolved: its end, and trial << 28 minus its first position (the key of
  // a one-pair record of the trial is this plus its position)
  int32_t t_end;
  uint32_t t_key;
  // positives left in the ring (fewer than 32), the lane's one of them, and the step they began in
  uint32_t left;
  uint32_t keep, keep_q;
  int32_t left_c0;
  // the group of positives whose rank-directory words are in flight
  uint32_t pd_n, pd_id;
  int32_t pd_pos;
  uint2 pd_rd;
};

// The ids of step c0: positions c0 + 8 lane .. c0 + 8 lane + 7.
__device__ __forceinline__ Ids8 gather_load(const GatherTile& g, int32_t c0, uint32_t lane) {
  Ids8 v;
#pragma unroll
  for (int j = 0; j < 8; ++j) v.e[j] = 0u;
  const int32_t i0 = c0 + 8 * static_cast<int32_t>(lane);
  if (i0 < g.span) v = ld_ids(g.ids + i0);
  return v;
}

// Finishes the group in flight (warp-wide): an event that is a member has its
// record appended to the tile's records, in lane order.
template <class Shared>
__device__ __forceinline__ void gather_complete(const GatherParams& p, const Shared& ws, GatherTile& g,
                                                uint32_t lane) {
  if (g.pd_n == 0u) return;
  const bool valid = lane < g.pd_n;
  // the word's bits up to the event's, the event's in the sign
  const uint32_t upto = __funnelshift_l(0u, g.pd_rd.x, ~g.pd_id);
  const bool hit = valid && static_cast<int32_t>(upto) < 0;
  uint32_t key = g.t_key + static_cast<uint32_t>(g.pd_pos);
  if (__any_sync(0xffffffffu, valid && g.pd_pos >= g.t_end)) {
    // a later trial: the last t with off[t] <= pos (off is padded with INT32_MAX)
    int t = (ws.off[4] <= g.pd_pos) ? 4 : 0;
    t += (ws.off[t + 2] <= g.pd_pos) ? 2 : 0;
    t += (ws.off[t + 1] <= g.pd_pos) ? 1 : 0;
    const uint32_t tk = (static_cast<uint32_t>(t) << kRecTrialShift) - static_cast<uint32_t>(ws.off[t]);
    key = tk + static_cast<uint32_t>(g.pd_pos);
    g.t_end = __shfl_sync(0xffffffffu, ws.off[t + 1], g.pd_n - 1u);
    g.t_key = __shfl_sync(0xffffffffu, tk, g.pd_n - 1u);
  }
  const uint32_t below = __popc(upto) - 1u, y = g.pd_rd.y;
  uint32_t ps = y + below;
  if (hit && (y & kRankSlots)) {  // the word holds an event with several pairs
    if ((y & kRankTwo) == kRankTwo) {
      const uint32_t two = (y >> kRankTwoShift) & 31u, bit = g.pd_id & 31u;
      ps = (y & kRankBaseMask) + below + (bit > two ? 1u : 0u);
      key += (bit == two ? 1u : 0u) << kRecCntShift;
    } else {
      const uint32_t slot = (y & kRankSlotMask) + below;
      ps = __ldg(&p.slot_start[slot]);
      key += (__ldg(&p.slot_start[slot + 1]) - ps - 1u) << kRecCntShift;
    }
  }
  const uint32_t hm = __ballot_sync(0xffffffffu, hit);
  if (hit) g.out[g.nout + __popc(hm & ((1u << lane) - 1u))] = make_uint2(key, ps);
  g.nout += __popc(hm);
}

// Puts a group of n positives in flight (lane < n: event id, position).
__device__ __forceinline__ void gather_launch(const GatherParams& p, GatherTile& g, uint32_t n, uint32_t id,
                                              int32_t pos, uint32_t lane) {
  g.pd_n = n;
  g.pd_id = id;
  g.pd_pos = pos;
  g.pd_rd = lane < n ? __ldg(&p.rankdir[id >> 5]) : make_uint2(0u, 0u);
}

// One step of 256 YET positions: filter, append the positives to the ring in
// YET order, then for every 32 of the ring finish the group in flight and put
// the next in flight; fewer than 32 stay for the next step.
// kSub: the catalogue has at most twice filt_words words, and word w folds
// onto min(w, w - filt_words) (unsigned); otherwise filt_words is a power of
// two and w folds onto w & (filt_words - 1).  fsel is filt_words or the mask.
template <bool kSub, bool kPacked>
__device__ __forceinline__ void gather_step(const GatherParams& p, const uint32_t* __restrict__ filt, uint32_t fsel,
                                            GatherShared<kPacked>& ws, GatherTile& g, int32_t c0, uint32_t lane,
                                            const Ids8& ids) {
  // 1. filter: bit j of m is position 8 lane + j's (the shift count of a funnel shift is taken mod 32)
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t wi = ids.e[j] >> 5;
    const uint32_t w = filt[kSub ? min(wi, wi - fsel) : (wi & fsel)];
    m = __funnelshift_r(m, __funnelshift_r(w, w, ids.e[j]), 1);
  }
  m >>= 24;
  const int32_t first = c0 + 8 * static_cast<int32_t>(lane);
  if (c0 == 0 || c0 + 256 > g.span) {
    // positions before the tile's first event and from its end on
    const int32_t lo = g.lead - first, hi = g.span - first;
    const uint32_t below = lo > 0 ? (lo < 8 ? (1u << lo) - 1u : 0xFFu) : 0u;
    const uint32_t upto = hi > 0 ? (hi < 8 ? (1u << hi) - 1u : 0xFFu) : 0u;
    m &= upto & ~below;
  }
  auto entry = [&](uint32_t i, uint32_t* v, uint32_t* q) {
    *v = ws.ring[i];
    if constexpr (!kPacked) *q = ws.ring_q[i];
  };
  auto send = [&](uint32_t v, uint32_t q, uint32_t k) {
    gather_complete(p, ws, g, lane);
    if constexpr (kPacked) {
      const int32_t last = c0 + 255;
      gather_launch(p, g, k, v >> kPosBits,
                    last - static_cast<int32_t>((static_cast<uint32_t>(last) - v) & ((1u << kPosBits) - 1u)), lane);
    } else {
      gather_launch(p, g, k, v, c0 + static_cast<int32_t>(q), lane);
    }
  };
  // 2. places in the ring: the lanes' counts summed from ballots of their bits (no shuffles, which share
  // the shared-memory pipe that bounds the kernel)
  const uint32_t cnt = __popc(m), lt = (1u << lane) - 1u;
  const uint32_t b0 = __ballot_sync(0xffffffffu, cnt & 1u), b1 = __ballot_sync(0xffffffffu, cnt & 2u),
                 b2 = __ballot_sync(0xffffffffu, cnt & 4u), b3 = __ballot_sync(0xffffffffu, cnt & 8u);
  if ((b0 | b1 | b2 | b3) != 0u) {
    uint32_t at = g.left + __popc(b0 & lt) + 2u * __popc(b1 & lt) + 4u * __popc(b2 & lt) + 8u * __popc(b3 & lt);
    if (g.left == 0u) g.left_c0 = c0;
    uint32_t n = g.left + __popc(b0) + 2u * __popc(b1) + 4u * __popc(b2) + 8u * __popc(b3);
    const uint32_t field = static_cast<uint32_t>(first) & ((1u << kPosBits) - 1u);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (m & (1u << j)) {
        if constexpr (kPacked) {
          ws.ring[at] = (ids.e[j] << kPosBits) + (field + j);
        } else {
          ws.ring[at] = ids.e[j];
          ws.ring_q[at] = static_cast<uint8_t>(8u * lane + j);
        }
        ++at;
      }
    __syncwarp();
    // 3. whole groups
    uint32_t r0 = 0u;
    uint32_t v = g.keep, q = g.keep_q;
    if (lane >= g.left) entry(lane, &v, &q);
    while (n >= 32u) {
      send(v, q, 32u);
      r0 += 32u;
      n -= 32u;
      entry(r0 + lane, &v, &q);  // past the last entry: a stale word that no group takes
      g.left_c0 = c0;
    }
    g.left = n;
    g.keep = v;
    g.keep_q = q;
    __syncwarp();
  }
  // 4. a packed position is told from its low bits while it lies within 2^kPosBits of the step's end, a position
  // in the step only in the step itself
  if (g.left > 0u && (!kPacked || c0 - g.left_c0 >= (1 << kPosBits) - 768)) {
    send(g.keep, g.keep_q, g.left);
    g.left = 0u;
  }
}

}  // namespace

template <bool kSub, bool kPacked>
__global__ void __launch_bounds__(kGatherThreads, 1) k_gather(const GatherParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Shared = GatherShared<kPacked>;
  Shared* gw = reinterpret_cast<Shared*>(smem_raw);
  uint32_t* filt = reinterpret_cast<uint32_t*>(gw + (kGatherThreads / 32));
  const uint32_t lane = lane_id();
  Shared& ws = gw[threadIdx.x >> 5];
  const uint32_t fsel = kSub ? static_cast<uint32_t>(p.filt_words) : static_cast<uint32_t>(p.filt_words) - 1u;

  for (int w = threadIdx.x; w < p.filt_words; w += blockDim.x) {
    uint32_t v = 0;
    for (int64_t k = w; k < p.n_words; k += p.filt_words) v |= p.rankdir[k].x;
    filt[w] = v;
  }
  __syncthreads();

  for (;;) {
    int64_t tile = 0;
    if (lane == 0) tile = static_cast<int64_t>(atomicAdd(p.queue, 1ull));
    tile = __shfl_sync(0xffffffffu, tile, 0);
    if (tile >= p.n_tiles) break;
    const int64_t ta = p.t_begin + tile * p.tile_trials;
    const int64_t tb = (ta + p.tile_trials < p.t_end) ? ta + p.tile_trials : p.t_end;
    const int ntr = static_cast<int>(tb - ta);
    const int64_t ea = __ldg(&p.off[ta]);
    GatherTile g;
    g.lead = static_cast<int32_t>(ea & 7);
    if (lane < 16)
      ws.off[lane] = (lane <= static_cast<uint32_t>(ntr))
                         ? static_cast<int32_t>(__ldg(&p.off[ta + lane]) - ea) + g.lead
                         : INT32_MAX;
    __syncwarp();
    g.span = ws.off[ntr];
    g.ids = p.ids + (ea & ~int64_t(7));
    g.out = p.ev_buf + (ea - p.e0);
    g.nout = 0;
    g.t_end = g.lead;  // the first group finds its trial
    g.t_key = 0u;
    g.left = 0u;
    g.keep = g.keep_q = 0u;
    g.left_c0 = 0;
    g.pd_n = 0u;
    // three steps of ids in registers, two of them in flight while one is filtered;
    // unrolled by three so that no register of a load in flight is ever moved
    Ids8 a = gather_load(g, 0, lane), b = gather_load(g, 256, lane), c;
    for (int32_t c0 = 0; c0 < g.span; c0 += 768) {
      c = gather_load(g, c0 + 512, lane);
      gather_step<kSub, kPacked>(p, filt, fsel, ws, g, c0, lane, a);
      if (c0 + 256 >= g.span) break;
      a = gather_load(g, c0 + 768, lane);
      gather_step<kSub, kPacked>(p, filt, fsel, ws, g, c0 + 256, lane, b);
      if (c0 + 512 >= g.span) break;
      b = gather_load(g, c0 + 1024, lane);
      gather_step<kSub, kPacked>(p, filt, fsel, ws, g, c0 + 512, lane, c);
    }
    gather_complete(p, ws, g, lane);
    if (g.left > 0u) {  // the last positives: within 2^kPosBits of the last step's end
      const int32_t last = ((g.span - 1) | 255);
      gather_launch(p, g, g.left, g.keep >> kPosBits,
                    last - static_cast<int32_t>((static_cast<uint32_t>(last) - g.keep) & ((1u << kPosBits) - 1u)), lane);
      gather_complete(p, ws, g, lane);
    }
    if (lane == 0) p.tile_cnt[tile] = g.nout;
    __syncwarp();
  }
}

cudaError_t launch_gather(const GatherParams& p, int grid, size_t smem, cudaStream_t s) {
  const bool sub = p.n_words <= 2 * static_cast<int64_t>(p.filt_words);
  auto launch = [&](auto kernel) -> cudaError_t {
    // (the limit belongs to the function: the most that any call asks for, as contexts on other threads
    // launch it too)
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 kGatherSmemBudget);
    if (err != cudaSuccess) return err;
    kernel<<<grid, kGatherThreads, smem, s>>>(p);
    return cudaGetLastError();
  };
  if (p.catalogue > kPackedCatalogue) return sub ? launch(k_gather<true, false>) : launch(k_gather<false, false>);
  return sub ? launch(k_gather<true, true>) : launch(k_gather<false, true>);
}

namespace {

constexpr int kQueue = 64;         // multi-ELT events queued per warp
constexpr uint32_t kDefCur = 1u;   // deferred event of the open tile
constexpr uint32_t kDefLast = 2u;  // last deferred event of its trial

struct LossWarp {
  float2 acc[kWarpTrials][32];  // per trial and lane: double-float sum of the lane's occurrence losses
  uint2 mq[kQueue];             // queued multi-ELT events (event records)
  uint32_t mqi[kQueue];         //   their places in the tile's records (per-event output)
  uint32_t d_key[32];           // deferred events: record
  uint32_t d_ps[32];            //   first pair
  int64_t d_o[32];              //   trial (output index)
  int64_t d_idx[32];            //   event buffer entry of the record (per-event output)
  uint32_t d_fl[32];            //   kDefCur | kDefLast
  float d_O[32];                //   occurrence loss, once resolved
  double Sd[kWarpTrials];       // sums of the deferred occurrence losses resolved while the tile is open
  unsigned long long hits[kWarpTrials];
  unsigned long long hash[kWarpTrials];
  unsigned long long n_nc, n_slow;  // non-converged Halley pairs, Halley events
};

// (hi, lo) + (hi2, lo2) in double-float arithmetic (TwoSum, then renormalise).
__device__ __forceinline__ void df_add(float& hi, float& lo, float hi2, float lo2) {
  const float s = hi + hi2;
  const float bb = s - hi;
  const float err = (hi - (s - bb)) + (hi2 - bb);
  const float e = err + lo + lo2;
  hi = s + e;
  lo = e - (hi - s);
}

// The table argument t = Phi^-1(z) of pair `pi` of an ELT record of kind
// `kind` (Beta or BetaC) in occurrence (trial, k); false when t lies beyond
// the tables' range (only a combined normal can).
__device__ __forceinline__ bool pair_normal(const LossParams& p, uint32_t kind, uint32_t elt, uint32_t pi,
                                            int64_t trial, uint32_t k, float* t) {
  if (kind == kKindBetaC) {
    *t = correlated_normal(p.rk, trial, k, elt, p.pw[pi]);
    return fabsf(*t) <= kTabT1f;
  }
  *t = normcdfinvf(philox_uniform_rk(p.rk, trial, k, elt));
  return true;
}

// Loss after ELT terms of pair `pi`, for the table path; returns false when
// the pair needs the Halley iteration.
__device__ __forceinline__ bool pair_fast(const LossParams& p, const Pair& pr, uint32_t pi, int64_t trial, uint32_t k,
                                          float* out) {
  const uint32_t kind = pair_kind(pr.meta);
  const uint32_t pos = pair_pos(pr.meta);
  float loss = pr.mu;
  if (kind == kKindZero) {
    loss = 0.0f;
  } else if (!p.primary_only && kind_is_beta(kind)) {
    if (p.newton_only || !pair_tab_exact(pr.meta)) return false;
    float t;
    if (!pair_normal(p, kind, static_cast<uint32_t>(p.elt_id[pos]), pi, trial, k, &t)) return false;
    const bool fine = pair_fine(pr.meta);
    const float4* tb = fine ? p.tabf[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabFineStride
                            : p.tab[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabNodes;
    loss = pr.max_l * tab_quantile_t(tb, t, fine);
  }
  *out = p.t_share[pos] * clamp_terms_f(loss, p.t_ret[pos], p.t_lim[pos]);
  return true;
}

__device__ __noinline__ float pair_slow(const LossParams& p, const Pair& pr, uint32_t pi, int64_t trial, uint32_t k,
                                        unsigned long long* nc) {
  const uint32_t pos = pair_pos(pr.meta);
  float v;
  if (pair_fast(p, pr, pi, trial, k, &v)) return v;
  const uint32_t elt = static_cast<uint32_t>(p.elt_id[pos]);
  const bool fine = pair_fine(pr.meta);
  const float4* tab = fine ? p.tabf[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabFineStride
                           : p.tab[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabNodes;
  BetaSolveStats st;
  float x;
  if (pair_kind(pr.meta) == kKindBetaC) {
    // z = Phi(v) and 1 - z = Phi(-v), each directly
    const float t = correlated_normal(p.rk, trial, k, elt, p.pw[pi]);
    x = pair_quantile_newton_zc(pr, normcdff(t), normcdff(-t), p.newton_only ? -1.0f : tab_quantile_t(tab, t, fine),
                                &st);
  } else {
    const float z = philox_uniform_rk(p.rk, trial, k, elt);
    x = pair_quantile_newton(pr, z, p.newton_only ? -1.0f : tab_quantile(tab, z, fine), &st);
  }
  if (!st.converged) ++*nc;
  return p.t_share[pos] * clamp_terms_f(pr.max_l * x, p.t_ret[pos], p.t_lim[pos]);
}

// Resolve the warp's deferred events (all lanes call it): lane i computes the
// occurrence loss of entry i, then lane 0 adds them in list order.  A trial's
// deferred losses form their own FP64 sum, in event order, so where the list
// is flushed does not change any result: entries of the open tile go to its
// shared sums, older ones to def_acc, and the last one of a trial finishes
// its year loss.  kEmit: also stores each entry's occurrence loss beside its
// record (per-event output).
template <bool kEmit>
__device__ __noinline__ void resolve_deferred(const LossParams& p, LossWarp& ws, int nd) {
  const uint32_t lane = lane_id();
  float O = 0.0f;
  unsigned long long nc_l = 0;
  unsigned long long* nc = &nc_l;
  if (lane < static_cast<uint32_t>(nd)) {
    const uint32_t key = ws.d_key[lane];
    const uint32_t k = key & kRecKMask;
    const uint32_t cnt = ((key >> kRecCntShift) & kRecCntMask) + 1u;
    const int64_t t = p.t_begin + ws.d_o[lane];
    float G = 0.0f;
    for (uint32_t j = 0; j < cnt; ++j) G += pair_slow(p, p.pairs[ws.d_ps[lane] + j], ws.d_ps[lane] + j, t, k, nc);
    O = clamp_terms_f(G, p.occ_r, p.occ_l);
    if constexpr (kEmit) p.occ[ws.d_idx[lane]] = O;
  }
  const uint32_t nc_w = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(nc_l));
  ws.d_O[lane] = O;
  __syncwarp();
  if (lane == 0) {
    ws.n_nc += nc_w;
    ws.n_slow += static_cast<unsigned long long>(nd);
    double acc = 0.0;
    bool open = false;  // acc holds def_acc of the current run's trial
    for (int i = 0; i < nd; ++i) {
      const float Oi = ws.d_O[i];
      const uint32_t fl = ws.d_fl[i];
      const int64_t o = ws.d_o[i];
      if (fl & kDefCur) {
        ws.Sd[ws.d_key[i] >> kRecTrialShift] += static_cast<double>(Oi);
        continue;
      }
      if (!open) {
        acc = p.def_acc[o];
        open = true;
      }
      acc += static_cast<double>(Oi);
      if (fl & kDefLast) {
        p.ylt[o] = clamp_terms_d(p.ylt[o] + acc, p.agg_r, p.agg_l);
        open = false;
      } else if (i + 1 == nd || ws.d_o[i + 1] != o) {
        p.def_acc[o] = acc;
        open = false;
      }
    }
  }
  __syncwarp();
}

}  // namespace

namespace {

// Appends this lane's event to the deferred list when `defer` (warp-wide call;
// events are listed in lane order), resolving the list first when it is full.
// Returns the new length of the list.  `idx` (kEmit) is the record's event
// buffer entry.
template <bool kEmit>
__device__ __forceinline__ int defer_events(const LossParams& p, LossWarp& ws, int nd, bool defer, uint2 r,
                                            int64_t o, int64_t idx) {
  const uint32_t dmask = __ballot_sync(0xffffffffu, defer);
  if (dmask == 0) return nd;
  if (nd + __popc(dmask) > 32) {
    resolve_deferred<kEmit>(p, ws, nd);
    nd = 0;
  }
  if (defer) {
    const int at = nd + __popc(dmask & ((1u << lane_id()) - 1u));
    ws.d_key[at] = r.x;
    ws.d_ps[at] = r.y;
    ws.d_o[at] = o;
    ws.d_fl[at] = kDefCur;
    if constexpr (kEmit) ws.d_idx[at] = idx;
  }
  __syncwarp();
  return nd + __popc(dmask);
}

// Adds an occurrence loss to the lane's double-float sum of trial tl.
__device__ __forceinline__ void acc_add(LossWarp& ws, uint32_t tl, float O) {
  float2 a = ws.acc[tl][lane_id()];
  df_add(a.x, a.y, O, 0.0f);
  ws.acc[tl][lane_id()] = a;
}

// The layer's ELTs by position, in shared memory (one array per field, so that
// lanes reading different ELTs hit different banks).
struct EltShared {
  const float4* tab[32];
  const float4* tabf[32];
  uint32_t elt_id[32];
  float ret[32], lim[32], share[32];
};

// A pair's loss between its two halves: known (kLossKnown: a), or from a table
// interval (kLossTable: a = max_l, s the place in the interval n0, n1), or by
// the Halley iteration (kLossSlow).
enum : uint32_t { kLossKnown = 0, kLossTable = 1, kLossSlow = 2 };
struct PairEval {
  uint32_t mode, pos;  // pos: the pair's ELT position
  float a, s;
  float4 n0;
  float2 n1;
};

// The first half, for lanes with `in`: the pair's normal and the loads of its
// table interval.  Callers put what they have to do for the next pairs between
// the halves, so that the loads are not waited for.
__device__ __forceinline__ PairEval pair_begin(const LossParams& p, const EltShared& es, LossWarp& ws, bool in,
                                               const PairHot& h, uint32_t pi, int64_t ta, uint32_t key, bool diag) {
  PairEval e{kLossKnown, pair_pos(h.meta), 0.0f, 0.0f, make_float4(0.0f, 0.0f, 0.0f, 0.0f), make_float2(0.0f, 0.0f)};
  if (in) {
    const uint32_t tl = key >> kRecTrialShift, k = key & kRecKMask;
    const uint32_t kind = pair_kind(h.meta);
    e.a = kind == kKindZero ? 0.0f : h.mu;
    if (!p.primary_only && kind_is_beta(kind)) {
      float t;
      if (p.newton_only || !pair_tab_exact(h.meta) || !pair_normal(p, kind, es.elt_id[e.pos], pi, ta + tl, k, &t)) {
        e.mode = kLossSlow;
      } else {
        const bool fine = pair_fine(h.meta);
        const TabPlace at = tab_place(t, fine);
        const float4* node = (fine ? es.tabf[e.pos] : es.tab[e.pos]) + h.node + at.i;
        e.mode = kLossTable;
        e.a = h.max_l;
        e.s = at.s;
        e.n0 = __ldg(node);
        e.n1 = __ldg(reinterpret_cast<const float2*>(node + 1) + 1);
      }
    }
    if (diag) {
      const uint32_t elt = es.elt_id[e.pos];
      atomicAdd(&ws.hits[tl], 1ull);
      atomicAdd(&ws.hash[tl], static_cast<unsigned long long>(fmix64((static_cast<uint64_t>(k) << 32) | elt)));
    }
  }
  return e;
}

// The second half: the pair's loss after ELT terms (meaningless for kLossSlow).
__device__ __forceinline__ float pair_end(const EltShared& es, const PairEval& e) {
  float loss = e.a;
  if (e.mode == kLossTable) loss = e.a * tab_value(e.s, e.n0, e.n1);
  return es.share[e.pos] * clamp_terms_f(loss, es.ret[e.pos], es.lim[e.pos]);
}

// A window's second half: the pairs' losses, a segmented sum per event (pairs
// in layer order), the occurrence terms at each event's last lane.  rec
// (kEmit): the lane's event's record's place in the tile.  Returns the deferred
// list's length.
template <bool kEmit>
__device__ __forceinline__ int window_end(const LossParams& p, const EltShared& es, LossWarp& ws, int nd,
                                          const PairWindow& w, const PairEval& e, int64_t ta, int64_t rb,
                                          uint32_t rec) {
  const uint32_t q = lane_id();
  const uint32_t ecnt = ((w.ex >> kRecCntShift) & kRecCntMask) + 1u;
  const uint32_t etl = w.ex >> kRecTrialShift;
  float L = pair_end(es, e);
  // segmented inclusive sum within each event's lanes
#pragma unroll
  for (uint32_t d = 1; d < 32; d <<= 1) {
    const float o = __shfl_up_sync(0xffffffffu, L, d);
    if (q >= w.epre + d) L += o;
  }
  const uint32_t smask = __ballot_sync(0xffffffffu, e.mode == kLossSlow);
  const bool end = q < w.np && q == w.epre + ecnt - 1u;
  const bool seg_slow = ((smask >> w.epre) & (0xffffffffu >> (31u - (q - w.epre)))) != 0u;
  if (end && !seg_slow) {
    const float O = clamp_terms_f(L, p.occ_r, p.occ_l);
    acc_add(ws, etl, O);
    if constexpr (kEmit) p.occ[rb + rec] = O;
  }
  return defer_events<kEmit>(p, ws, nd, end && seg_slow, make_uint2(w.ex, w.ey), ta + etl - p.t_begin, rb + rec);
}

// The queued multi-ELT events, in windows.  Returns (deferred list length,
// pairs processed).  kEmit: the occurrence losses also go beside the records
// (the tile's records start at event buffer entry rb).
template <bool kEmit>
__device__ __forceinline__ int2 process_multi(const LossParams& p, const EltShared& es, LossWarp& ws, int nd, int nq,
                                              int64_t ta, bool diag, int64_t rb) {
  const uint32_t q = lane_id();
  int n_pairs = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < nq;) {
    const int ie = i0 + static_cast<int>(q);
    const uint2 r = (ie < nq) ? ws.mq[ie] : make_uint2(0u, 0u);
    const PairWindow w = make_window(r, (ie < nq) ? ((r.x >> kRecCntShift) & kRecCntMask) + 1u : 0u);
    PairHot h{0.0f, 0.0f, kKindZero << kMetaKindShift, 0u};
    if (q < w.np) h = p.hot[w.ey + (q - w.epre)];
    n_pairs += static_cast<int>(w.np);
    const PairEval e = pair_begin(p, es, ws, q < w.np, h, w.ey + (q - w.epre), ta, w.ex, diag);
    uint32_t rec = 0u;
    if constexpr (kEmit)
      if (q < w.np) rec = ws.mqi[i0 + w.ev];
    nd = window_end<kEmit>(p, es, ws, nd, w, e, ta, rb, rec);
    i0 += w.n_take;
  }
  __syncwarp();
  return make_int2(nd, n_pairs);
}

// One stage of the reduce-scatter of kWarpTrials double-float values over the
// warp: lanes with bit (4 HALF) clear keep values 0..HALF-1, the others
// HALF..2 HALF-1, each adding its partner's copy of the values it keeps.
template <int HALF>
__device__ __forceinline__ void reduce_scatter_stage(float (&h)[kWarpTrials], float (&l)[kWarpTrials], uint32_t lane) {
  constexpr int d = 4 * HALF;
  const bool up = (lane & d) != 0;
#pragma unroll
  for (int j = 0; j < HALF; ++j) {
    const float sh = up ? h[j] : h[j + HALF], sl = up ? l[j] : l[j + HALF];
    float kh = up ? h[j + HALF] : h[j], kl = up ? l[j + HALF] : l[j];
    df_add(kh, kl, __shfl_xor_sync(0xffffffffu, sh, d), __shfl_xor_sync(0xffffffffu, sl, d));
    h[j] = kh;
    l[j] = kl;
  }
}

}  // namespace

// k_losses: each warp takes tiles and sums their events' occurrence losses: per
// pair the Philox uniform, the inverse Beta through the record's quantile table
// and the ELT terms, per event the occurrence terms and a double-float add into
// the lane's sum for the event's trial.  At the end of the tile one
// reduce-scatter over the lanes turns the per-lane sums into the trials' sums.
// kEmit (per-event output) also stores each hit event's occurrence loss beside
// its record.
//
// !kWindows: a lane per event record (the records two rounds ahead and the hot
// pair records one round ahead are in flight); events with several pairs are
// queued and processed in windows of 32 pairs with a segmented sum.  For layers
// where nearly all hit events have one pair.
// kWindows: every event in windows of up to 32 pairs of whole events, a lane
// per pair, laid out from the records as they come.
//
// Bound by the latency of the table intervals (random 24-byte reads, past L1)
// with 24 warps an SM, then by L1's rate of misses: so each pair is computed in
// two halves, its interval's loads and its loss, and the next round or window
// is prepared between them.  1M trials of 75 pairs, a lane per event: 1,005 us
// (1,030 with the loads waited for); 100,003 trials of 750 pairs over 30 ELTs of
// 100,000 events, in windows: 1,140 us (1,740 with a lane per event and the
// events of several pairs, most of them there, queued).
template <bool kEmit, bool kWindows>
__global__ void __launch_bounds__(kLossThreads, kLossBlocksPerSm) k_losses(const LossParams p) {
  __shared__ LossWarp lw[kLossThreads / 32];
  __shared__ EltShared es;
  const uint32_t lane = lane_id();
  LossWarp& ws = lw[threadIdx.x >> 5];
  if (threadIdx.x < 32) {
    const int i = static_cast<int>(threadIdx.x);
    const bool in = i < p.n_elts;
    es.tab[i] = in ? p.tab[i] : nullptr;
    es.tabf[i] = in ? p.tabf[i] : nullptr;
    es.elt_id[i] = in ? static_cast<uint32_t>(p.elt_id[i]) : 0u;
    es.ret[i] = in ? p.t_ret[i] : 0.0f;
    es.lim[i] = in ? p.t_lim[i] : 0.0f;
    es.share[i] = in ? p.t_share[i] : 0.0f;
  }
  __syncthreads();
  const bool diag = (p.diag_hits != nullptr) || (p.diag_hash != nullptr);
  const uint32_t lt_mask = (1u << lane) - 1u;
  int nd = 0;  // deferred events listed; the list outlives tiles so that resolving keeps the lanes busy
  uint32_t n_pairs = 0;
  if (lane == 0) {
    ws.n_nc = 0ull;
    ws.n_slow = 0ull;
  }

  for (;;) {
    int64_t tile = 0;
    if (lane == 0) tile = static_cast<int64_t>(atomicAdd(&p.counters[0], 1ull));
    tile = __shfl_sync(0xffffffffu, tile, 0);
    if (tile >= p.n_tiles) break;
    const int64_t ta = p.t_begin + tile * p.tile_trials;
    const int64_t tb = (ta + p.tile_trials < p.t_end) ? ta + p.tile_trials : p.t_end;
    const int ntr = static_cast<int>(tb - ta);
    const int64_t rb = __ldg(&p.off[ta]) - p.e0;  // the tile's first event buffer entry
    const uint2* recs = p.ev_buf + rb;
    const uint32_t n = __ldg(&p.tile_cnt[tile]);
#pragma unroll
    for (int t = 0; t < kWarpTrials; ++t) ws.acc[t][lane] = make_float2(0.0f, 0.0f);
    if (lane < static_cast<uint32_t>(ntr)) {
      ws.Sd[lane] = 0.0;
      ws.hits[lane] = 0ull;
      ws.hash[lane] = 0ull;
    }
    __syncwarp();
    if constexpr (!kWindows) {
      int nq = 0;
      // pipeline: r1 = records of the next round, r0/h0 = this round's record and hot pair
      uint2 r0 = (lane < n) ? __ldcs(recs + lane) : make_uint2(0u, 0u);
      uint2 r1 = (32 + lane < n) ? __ldcs(recs + 32 + lane) : make_uint2(0u, 0u);
      PairHot h0{0.0f, 0.0f, kKindZero << kMetaKindShift, 0u};
      if (lane < n && ((r0.x >> kRecCntShift) & kRecCntMask) == 0u) h0 = p.hot[r0.y];
      for (uint32_t base = 0;;) {
#pragma unroll 1
        for (; base < n && nq <= kQueue - 32; base += 32) {
          const uint2 r = r0;
          const bool valid = base + lane < n;
          const uint32_t cnt = ((r.x >> kRecCntShift) & kRecCntMask) + 1u;
          const bool single = valid && cnt == 1u;
          const PairEval e = pair_begin(p, es, ws, single, h0, r.y, ta, r.x, diag);
          // the next round's loads and the queue, while the table interval comes
          r0 = r1;
          if (base + 64 + lane < n) r1 = __ldcs(recs + base + 64 + lane);
          if (base + 32 + lane < n && ((r0.x >> kRecCntShift) & kRecCntMask) == 0u) h0 = p.hot[r0.y];
          const uint32_t mmask = __ballot_sync(0xffffffffu, valid && cnt > 1u);
          if (mmask) {
            if (valid && cnt > 1u) {
              ws.mq[nq + __popc(mmask & lt_mask)] = r;
              if constexpr (kEmit) ws.mqi[nq + __popc(mmask & lt_mask)] = base + lane;
            }
            nq += __popc(mmask);
          }
          const bool slow = single && e.mode == kLossSlow;
          if (single && !slow) {
            const float O = clamp_terms_f(pair_end(es, e), p.occ_r, p.occ_l);
            acc_add(ws, r.x >> kRecTrialShift, O);
            if constexpr (kEmit) p.occ[rb + base + lane] = O;
          }
          n_pairs += __popc(__ballot_sync(0xffffffffu, single));
          nd = defer_events<kEmit>(p, ws, nd, slow, r, ta + (r.x >> kRecTrialShift) - p.t_begin, rb + base + lane);
        }
        __syncwarp();
        if (nq > 0) {
          const int2 rv = process_multi<kEmit>(p, es, ws, nd, nq, ta, diag, rb);
          nd = rv.x;
          n_pairs += static_cast<uint32_t>(rv.y);
          nq = 0;
        }
        if (base >= n) break;
      }
    } else {
      // a window's table intervals are in flight while the next window is laid out, that one's hot records
      // while this one's sums are made, and the records after it meanwhile
      auto count_of = [](uint2 r, bool in) { return in ? ((r.x >> kRecCntShift) & kRecCntMask) + 1u : 0u; };
      uint2 r = (lane < n) ? __ldg(recs + lane) : make_uint2(0u, 0u);
      uint32_t next = 0u;  // the first record after the window
      PairWindow w;
      PairHot h;
      auto next_window = [&]() {
        w = make_window(r, count_of(r, next + lane < n));
        h = PairHot{0.0f, 0.0f, kKindZero << kMetaKindShift, 0u};
        if (lane < w.np) h = p.hot[w.ey + (lane - w.epre)];
        next += static_cast<uint32_t>(w.n_take);
        if (next + lane < n) r = __ldg(recs + next + lane);
      };
      next_window();
#pragma unroll 1
      while (w.np != 0u) {
        const PairEval e = pair_begin(p, es, ws, lane < w.np, h, w.ey + (lane - w.epre), ta, w.ex, diag);
        const PairWindow v = w;
        const uint32_t rec = next - static_cast<uint32_t>(w.n_take) + w.ev;
        n_pairs += w.np;
        next_window();
        nd = window_end<kEmit>(p, es, ws, nd, v, e, ta, rb, rec);
      }
    }
    __syncwarp();
    // ---- trials' sums: reduce-scatter of the per-lane double-float sums; lane
    // (b4 b3 b2 b1 b0) ends up holding trial 4 b4 + 2 b3 + b2
    float h8[kWarpTrials], l8[kWarpTrials];
#pragma unroll
    for (int t = 0; t < kWarpTrials; ++t) {
      const float2 a = ws.acc[t][lane];
      h8[t] = a.x;
      l8[t] = a.y;
    }
    reduce_scatter_stage<4>(h8, l8, lane);
    reduce_scatter_stage<2>(h8, l8, lane);
    reduce_scatter_stage<1>(h8, l8, lane);
#pragma unroll
    for (int d = 2; d > 0; d >>= 1) {
      const float h2 = __shfl_xor_sync(0xffffffffu, h8[0], d);
      const float l2 = __shfl_xor_sync(0xffffffffu, l8[0], d);
      df_add(h8[0], l8[0], h2, l2);
    }
    const uint32_t src = ((lane >> 2) & 1u) << 4 | ((lane >> 1) & 1u) << 3 | (lane & 1u) << 2;
    const float Sh = __shfl_sync(0xffffffffu, h8[0], src);
    const float Sl = __shfl_sync(0xffffffffu, l8[0], src);
    const double S = static_cast<double>(Sh) + static_cast<double>(Sl);
    // ---- tile end: a trial whose deferred events are all resolved is final; one
    // with events still listed keeps its table-path sum in ylt and its partial
    // deferred sum in def_acc until the last of them is resolved
    uint32_t pend = 0;
    {
      const bool cur = lane < static_cast<uint32_t>(nd) && (ws.d_fl[lane] & kDefCur);
      const uint32_t tl = cur ? (ws.d_key[lane] >> kRecTrialShift) : 0xFFu + lane;
      const uint32_t same = __match_any_sync(0xffffffffu, tl);
      if (cur) {
        pend = 1u << tl;
        ws.d_fl[lane] = (lane == 31u - __clz(same)) ? kDefLast : 0u;
      }
    }
    pend = __reduce_or_sync(0xffffffffu, pend);
    __syncwarp();
    if (lane < static_cast<uint32_t>(ntr)) {
      const int64_t o = ta + lane - p.t_begin;
      if ((pend >> lane) & 1u) {
        p.ylt[o] = S;
        p.def_acc[o] = ws.Sd[lane];
      } else {
        p.ylt[o] = clamp_terms_d(S + ws.Sd[lane], p.agg_r, p.agg_l);
      }
      if (p.diag_hits) p.diag_hits[o] = static_cast<int64_t>(ws.hits[lane]);
      if (p.diag_hash) p.diag_hash[o] = ws.hash[lane];
    }
    __syncwarp();
  }
  if (nd > 0) resolve_deferred<kEmit>(p, ws, nd);
  if (lane == 0) {
    const unsigned long long n_nc = ws.n_nc, n_slow = ws.n_slow;
    if (n_pairs) atomicAdd(&p.counters[1], static_cast<unsigned long long>(n_pairs));
    if (n_nc) atomicAdd(&p.counters[2], n_nc);
    if (n_slow) atomicAdd(&p.counters[3], n_slow);
  }
}

cudaError_t launch_losses(const LossParams& p, int grid, cudaStream_t s) {
  if (p.windows) {
    if (p.occ)
      k_losses<true, true><<<grid, kLossThreads, 0, s>>>(p);
    else
      k_losses<false, true><<<grid, kLossThreads, 0, s>>>(p);
  } else if (p.occ) {
    k_losses<true, false><<<grid, kLossThreads, 0, s>>>(p);
  } else {
    k_losses<false, false><<<grid, kLossThreads, 0, s>>>(p);
  }
  return cudaGetLastError();
}

}  // namespace ara
