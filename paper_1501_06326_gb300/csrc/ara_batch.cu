// Several layers in one pass (a batch): the losses kernel after k_gather has
// found, over the union of the batch's ELTs, the hit events of each tile.
//
// Each (event occurrence, ELT) loss after ELT terms (Philox uniform, inverse
// Beta through the record's quantile table, ELT terms; Section 3.3) is
// computed once and serves every layer of the batch that holds the ELT.  Per
// layer, the event's losses over the layer's ELTs are summed (Algorithm 1),
// the occurrence terms applied, and the occurrence loss is added to the
// layer's sum for the trial: a 64-bit fixed-point integer (each loss rounded
// to the layer's unit, about 2^-61 of its largest possible trial sum), so that
// the sum is exact in those units and independent of the order of the
// (atomic) additions.  The aggregate terms of each layer then give its year
// losses.  Three kernels do this with different work items (a lane per record
// over a tile or over one trial, or a lane per pair over a tile); they add the
// same fixed-point numbers and give the same results.
#include <cuda_runtime.h>

#include <cstdint>

#include "ara_batch.h"
#include "ara_window.cuh"

namespace ara {

namespace {

constexpr int kBatchQueue = 64;  // multi-ELT events queued per warp

struct BatchWarp {
  unsigned long long acc[kBatchLayers][32];  // per layer and lane: the lane's sum for its current trial (fixed point)
  unsigned long long (*tacc)[kWarpTrials];  // per layer and trial of the tile: the trial's sum (tiles only)
  uint32_t act[kWarpTrials];                 // per trial of the tile: the layers whose trials reach it
  uint2 mq[kBatchQueue];                     // queued multi-ELT events (records)
  float wl[32];                              // a window's pair losses
  unsigned long long wm[32];                 // a window's pairs: layers holding the pair's ELT
};

struct BatchShared {
  const float4* tab[kMaxIndexElts];
  const float4* tabf[kMaxIndexElts];
  uint32_t elt_id[kMaxIndexElts];
  float ret[kMaxIndexElts], lim[kMaxIndexElts], share[kMaxIndexElts];
  unsigned long long layers_of[kMaxIndexElts];
  float occ_r[kBatchLayers], occ_l[kBatchLayers];
  float scale[kBatchLayers];
  int64_t t_end[kBatchLayers];
};

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }

// O in a layer's fixed-point units: O * scale rounded to the nearest integer
// (ties to even).  O >= 0 is finite and scale a power of two, so the product is
// exact (or below one unit) and O * scale < 2^62 by the choice of scale.
__device__ __forceinline__ unsigned long long fixed_units(float O, float scale) {
  return __float2ull_rn(O * scale);
}

// The table argument t = Phi^-1(z) of pair `pi` (a record of kind Beta or
// BetaC) in occurrence (trial, k); false when t lies beyond the tables' range
// (only a combined normal can).
__device__ __forceinline__ bool batch_pair_normal(const BatchParams& p, uint32_t kind, uint32_t elt, uint32_t pi,
                                                  int64_t trial, uint32_t k, float* t) {
  if (kind == kKindBetaC) {
    *t = correlated_normal(p.rk, trial, k, elt, p.pw[pi]);
    return fabsf(*t) <= kTabT1f;
  }
  *t = normcdfinvf(philox_uniform_rk(p.rk, trial, k, elt));
  return true;
}

// Loss after ELT terms of pair `pi` by the Halley iteration: when the record's
// table is not exact, when a combined normal lies beyond the tables' range, or
// when the layers ask for it.
__device__ __noinline__ float pair_loss_slow(const BatchParams& p, const Pair& pr, uint32_t pi, int64_t trial,
                                             uint32_t k, unsigned long long* nc) {
  const uint32_t pos = pair_pos(pr.meta);
  const uint32_t elt = static_cast<uint32_t>(p.elt_id[pos]);
  const bool fine = pair_fine(pr.meta);
  const float4* tab = fine ? p.tabf[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabFineStride
                           : p.tab[pos] + static_cast<size_t>(pair_rec(pr.meta)) * kTabNodes;
  BetaSolveStats st;
  float x;
  if (pair_kind(pr.meta) == kKindBetaC) {
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

__device__ __forceinline__ float pair_loss_batch(const BatchParams& p, const BatchShared& bs, uint32_t pair_index,
                                                 int64_t trial, uint32_t k, unsigned long long* nc) {
  const PairHot h = p.hot[pair_index];
  const uint32_t kind = pair_kind(h.meta);
  const uint32_t pos = pair_pos(h.meta);
  float loss = h.mu;
  if (kind == kKindZero) {
    loss = 0.0f;
  } else if (!p.primary_only && kind_is_beta(kind)) {
    if (p.newton_only || !pair_tab_exact(h.meta))
      return pair_loss_slow(p, p.pairs[pair_index], pair_index, trial, k, nc);
    float t;
    if (!batch_pair_normal(p, kind, bs.elt_id[pos], pair_index, trial, k, &t))
      return pair_loss_slow(p, p.pairs[pair_index], pair_index, trial, k, nc);
    const bool fine = pair_fine(h.meta);
    const float4* tb = (fine ? bs.tabf[pos] : bs.tab[pos]) + h.node;
    loss = h.max_l * tab_quantile_t(tb, t, fine);
  }
  return bs.share[pos] * clamp_terms_f(loss, bs.ret[pos], bs.lim[pos]);
}

// Adds a layer's occurrence loss (from the event's loss sum G over the
// layer's ELTs) to the lane's fixed-point sum for its current trial.
__device__ __forceinline__ void add_occurrence(BatchWarp& ws, const BatchShared& bs, int layer, uint32_t lane,
                                               float G, uint32_t* dirty) {
  const float O = clamp_terms_f(G, bs.occ_r[layer], bs.occ_l[layer]);
  if (O > 0.0f) {
    ws.acc[layer][lane] += fixed_units(O, bs.scale[layer]);
    *dirty |= 1u << layer;
  }
}

// The same, straight into the trial's sum of the tile (events whose lane is
// not tracking their trial: the multi-ELT ones).
__device__ __forceinline__ void add_occurrence_trial(BatchWarp& ws, const BatchShared& bs, int layer, uint32_t tl,
                                                     float G) {
  const float O = clamp_terms_f(G, bs.occ_r[layer], bs.occ_l[layer]);
  if (O > 0.0f) atomicAdd(&ws.tacc[layer][tl], fixed_units(O, bs.scale[layer]));
}

// Moves the lane's sums of the layers in `dirty` into the tile's sums of
// trial tl.
__device__ __forceinline__ void flush_lane(BatchWarp& ws, uint32_t lane, uint32_t tl, uint32_t dirty) {
  for (uint32_t m = dirty; m; m &= m - 1u) {
    const int l = __ffs(m) - 1;
    atomicAdd(&ws.tacc[l][tl], ws.acc[l][lane]);
    ws.acc[l][lane] = 0ull;
  }
}

// A multi-ELT event with more pairs than a window holds, by one lane: for each
// layer it touches, its pair losses over the layer's ELTs summed in the pairs'
// order (each pair's loss recomputed per layer: such events are rare).
template <bool kPerTrial>
__device__ __noinline__ void batch_long_event(const BatchParams& p, const BatchShared& bs, BatchWarp& ws, uint2 r,
                                              int64_t ta, unsigned long long* nc) {
  const uint32_t cnt = ((r.x >> kRecCntShift) & kRecCntMask) + 1u;
  const uint32_t k = r.x & kRecKMask;
  const uint32_t tl = r.x >> kRecTrialShift;
  unsigned long long touched = 0ull;
  for (uint32_t j = 0; j < cnt; ++j) touched |= bs.layers_of[pair_pos(p.hot[r.y + j].meta)];
  for (unsigned long long m = touched & ws.act[tl]; m; m &= m - 1ull) {
    const int l = __ffsll(m) - 1;
    float G = 0.0f;
    for (uint32_t j = 0; j < cnt; ++j)
      if ((bs.layers_of[pair_pos(p.hot[r.y + j].meta)] >> l) & 1ull) G += pair_loss_batch(p, bs, r.y + j, ta + tl, k, nc);
    if (kPerTrial) {
      uint32_t unused = 0u;
      add_occurrence(ws, bs, l, lane_id(), G, &unused);
    } else {
      add_occurrence_trial(ws, bs, l, tl, G);
    }
  }
}

// The queued multi-ELT events of a tile, in windows of at most 32 pairs
// (one per lane): each pair's loss once, then for each layer the window's
// events touch, each event's last lane sums the event's pair losses of that
// layer from left to right (the pairs' canonical order), applies the
// occurrence terms and adds the result to its trial's sum.  A left-to-right
// sum does not change when pairs of other layers' ELTs are present, so an
// event's per-layer losses are the same in any batch.  Only the layers that
// reach the event's trial are served; a pair of none of them is not computed.
// kPerTrial: all events are of one trial, and the end lanes add into their own
// sums (no contention); else into the trial's sum of the tile.
template <bool kPerTrial>
__device__ __noinline__ uint32_t batch_multi(const BatchParams& p, const BatchShared& bs, BatchWarp& ws, int nq,
                                             int64_t ta, unsigned long long* nc) {
  const uint32_t q = lane_id();
  const uint32_t upto = 0xffffffffu >> (31u - q);  // lanes 0..q
  uint32_t n_pairs = 0;
  for (int i0 = 0; i0 < nq;) {
    const int ie = i0 + static_cast<int>(q);
    const uint2 r = (ie < nq) ? ws.mq[ie] : make_uint2(0u, 0u);
    const uint32_t cnt = (ie < nq) ? ((r.x >> kRecCntShift) & kRecCntMask) + 1u : 0u;
    if (__shfl_sync(0xffffffffu, cnt, 0) > 32u) {  // a long event first in line: by lane 0
      if (q == 0) batch_long_event<kPerTrial>(p, bs, ws, r, ta, nc);
      n_pairs += __shfl_sync(0xffffffffu, cnt, 0);
      __syncwarp();
      ++i0;
      continue;
    }
    uint32_t incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (q >= static_cast<uint32_t>(d)) incl += o;
    }
    const uint32_t pre = incl - cnt;
    const bool take = cnt != 0 && incl <= 32u;
    const int n_take = __popc(__ballot_sync(0xffffffffu, take));
    const uint32_t np = __shfl_sync(0xffffffffu, incl, n_take - 1);
    const uint32_t starts = __reduce_or_sync(0xffffffffu, take ? (1u << pre) : 0u);
    const uint32_t ev = static_cast<uint32_t>(__popc(starts & upto)) - 1u;  // lane q's event
    const uint32_t ex = __shfl_sync(0xffffffffu, r.x, ev);
    const uint32_t ey = __shfl_sync(0xffffffffu, r.y, ev);
    const uint32_t epre = __shfl_sync(0xffffffffu, pre, ev);
    const uint32_t ecnt = __shfl_sync(0xffffffffu, cnt, ev);
    const uint32_t etl = ex >> kRecTrialShift;
    float L = 0.0f;
    unsigned long long lm = 0ull;
    if (q < np) {
      lm = bs.layers_of[pair_pos(p.hot[ey + (q - epre)].meta)] & ws.act[etl];
      if (lm) L = pair_loss_batch(p, bs, ey + (q - epre), ta + etl, ex & kRecKMask, nc);
    }
    ws.wl[q] = L;
    ws.wm[q] = lm;
    n_pairs += np;
    const bool end = q < np && q == epre + ecnt - 1u;
    unsigned long long touched = lm;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) touched |= __shfl_xor_sync(0xffffffffu, touched, d);
    __syncwarp();
    for (unsigned long long m = touched; m; m &= m - 1ull) {
      const int l = __ffsll(m) - 1;
      if (end) {
        float G = 0.0f;
        for (uint32_t j = epre; j <= q; ++j)
          if ((ws.wm[j] >> l) & 1ull) G += ws.wl[j];
        if (kPerTrial) {
          uint32_t unused = 0u;
          add_occurrence(ws, bs, l, q, G, &unused);
        } else {
          add_occurrence_trial(ws, bs, l, etl, G);
        }
      }
    }
    __syncwarp();
    i0 += n_take;
  }
  __syncwarp();
  return n_pairs;
}

// First record in [0, n) whose trial is >= key (n if none), by the whole warp:
// each round probes 32 evenly spaced records and keeps the gap between the
// last probe below key and the first at or above it.
__device__ __forceinline__ int32_t first_record_of(const uint2* recs, int32_t n, uint32_t key, uint32_t lane) {
  int32_t lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const int32_t step = (hi - lo + 31) / 32;
    const int32_t pos = lo + static_cast<int32_t>(lane) * step;
    const bool ge = pos < hi && (__ldg(&recs[pos].x) >> kRecTrialShift) >= key;
    const uint32_t b = __ballot_sync(0xffffffffu, ge);
    if (b == 0u) {
      const int32_t probes = (hi - lo + step - 1) / step;  // positions lo + j step < hi
      lo += (probes - 1) * step + 1;
    } else {
      const int32_t f = __ffs(b) - 1;
      hi = lo + f * step;
      if (f > 0) lo += (f - 1) * step + 1;
    }
  }
  return lo;
}

}  // namespace

// One warp per item, the item's hit-event records two per lane per round
// (records two rounds ahead and single-ELT hot pairs one round ahead in
// flight); every lane keeps its own fixed-point sum per layer.
// kPerTrial = false: an item is a tile of up to kWarpTrials trials.  A lane's
//   records come in trial order, so its sums are for its current trial and
//   move into the tile's per-trial sums (shared-memory atomics) when the
//   trial changes.  Few records per trial fill the lanes this way.
// kPerTrial = true: an item is one trial of a tile (its records found by a
//   warp search), and the lanes' sums are added once at the item's end.
//   Many records per trial (many ELTs in the batch) keep the lanes busy, and
//   the lanes do not contend for the same sums.
// Multi-ELT events add into the per-trial sums directly.  At the item's end
// the aggregate terms of each layer give the year losses.  Both kinds add the
// same fixed-point numbers, so they give the same results.
template <bool kPerTrial>
__global__ void __launch_bounds__(kBatchThreads, kBatchBlocksPerSm) k_losses_batch(const BatchParams p) {
  __shared__ BatchWarp bw[kBatchThreads / 32];
  __shared__ BatchShared bs;
  // (one-trial items need none: a placeholder keeps the block within the shared-memory
  // carveout that leaves L1 its room)
  __shared__ unsigned long long tacc_all[kPerTrial ? 1 : kBatchThreads / 32][kPerTrial ? 1 : kBatchLayers][kWarpTrials];
  const uint32_t lane = lane_id();
  BatchWarp& ws = bw[threadIdx.x >> 5];
  if (lane == 0) ws.tacc = tacc_all[kPerTrial ? 0 : threadIdx.x >> 5];
  for (int i = threadIdx.x; i < kMaxIndexElts; i += blockDim.x) {
    const bool in = i < p.n_elts;
    bs.tab[i] = in ? p.tab[i] : nullptr;
    bs.tabf[i] = in ? p.tabf[i] : nullptr;
    bs.elt_id[i] = in ? static_cast<uint32_t>(p.elt_id[i]) : 0u;
    bs.ret[i] = in ? p.t_ret[i] : 0.0f;
    bs.lim[i] = in ? p.t_lim[i] : 0.0f;
    bs.share[i] = in ? p.t_share[i] : 0.0f;
    bs.layers_of[i] = in ? p.layers_of[i] : 0ull;
  }
  for (int i = threadIdx.x; i < kBatchLayers; i += blockDim.x) {
    bs.occ_r[i] = p.occ_r[i];
    bs.occ_l[i] = p.occ_l[i];
    bs.scale[i] = p.scale[i];
    bs.t_end[i] = i < p.n_layers ? p.layer_t_end[i] : 0;
  }
  __syncthreads();
  static_assert(kBatchLayers <= 32, "one lane per layer");
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int nl = p.n_layers;
  unsigned long long nc = 0ull;
  uint32_t n_pairs = 0;
  for (int l = 0; l < nl; ++l) ws.acc[l][lane] = 0ull;
  const int64_t n_items = kPerTrial ? p.n_tiles * p.tile_trials : p.n_tiles;

  // items are claimed one ahead, so that the claim's latency overlaps an item's work
  unsigned long long next = 0ull;
  if (lane == 0) next = atomicAdd(&p.counters[0], 1ull);
  for (;;) {
    const int64_t item = static_cast<int64_t>(__shfl_sync(0xffffffffu, next, 0));
    if (item >= n_items) break;
    if (lane == 0) next = atomicAdd(&p.counters[0], 1ull);
    const int64_t tile = kPerTrial ? item / p.tile_trials : item;
    const uint32_t tl0 = kPerTrial ? static_cast<uint32_t>(item % p.tile_trials) : 0u;  // the item's first trial
    const int64_t ta = p.t_begin + tile * p.tile_trials;
    const int ntr = static_cast<int>((ta + p.tile_trials < p.t_end) ? p.tile_trials : p.t_end - ta);
    if (kPerTrial && static_cast<int>(tl0) >= ntr) continue;
    const int t_lo = static_cast<int>(tl0);  // the item's (first) trial in the tile
    // per trial of the item, the layers whose trials reach it (all of them unless a layer ends early)
    uint32_t any = 0u;
#pragma unroll
    for (int t = 0; t < kWarpTrials; ++t) {
      if (kPerTrial && t != t_lo) continue;
      const uint32_t a =
          __ballot_sync(0xffffffffu, t < ntr && lane < static_cast<uint32_t>(nl) && ta + t < bs.t_end[lane]);
      if (lane == 0) ws.act[t] = a;
      any |= a;
    }
    if (!kPerTrial)
      for (int i = static_cast<int>(lane); i < nl * kWarpTrials; i += 32) ws.tacc[i / kWarpTrials][i % kWarpTrials] = 0ull;
    __syncwarp();
    const uint2* recs = p.ev_buf + (__ldg(&p.off[ta]) - p.e0);
    const int32_t n_tile = any ? static_cast<int32_t>(__ldg(&p.tile_cnt[tile])) : 0;
    // the item's records [beg, n) of the tile (records are in trial order)
    const int32_t beg = kPerTrial ? first_record_of(recs, n_tile, tl0, lane) : 0;
    const int32_t n = kPerTrial ? first_record_of(recs, n_tile, tl0 + 1, lane) : n_tile;
    if (kPerTrial) {  // each lane clears its own sums (conflict-free)
      __syncwarp();
      for (int l = 0; l < nl; ++l) ws.acc[l][lane] = 0ull;
    }
    uint32_t cur = tl0, dirty = 0u;  // the lane's current trial, and the layers its sums hold
    const uint32_t act0 = ws.act[t_lo];  // the item's layers (one trial)
    int nq = 0;
    // 64 records per round, two per lane (lane and 32 + lane), so that two table
    // reads are in flight per lane; the next round's records and single-ELT hot
    // pairs are loaded one round ahead
    uint2 rn[2];
    PairHot hn[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int32_t at = beg + 32 * j + static_cast<int32_t>(lane);
      rn[j] = (at < n) ? __ldcs(recs + at) : make_uint2(0u, 0u);
      hn[j] = PairHot{0.0f, 0.0f, kKindZero << kMetaKindShift, 0u};
      if (at < n && ((rn[j].x >> kRecCntShift) & kRecCntMask) == 0u) hn[j] = p.hot[rn[j].y];
    }
    for (int32_t base = beg; base < n; base += 64) {
      uint2 r[2];
      PairHot h[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        r[j] = rn[j];
        h[j] = hn[j];
        const int32_t at = base + 64 + 32 * j + static_cast<int32_t>(lane);
        if (at < n) rn[j] = __ldcs(recs + at);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int32_t at = base + 64 + 32 * j + static_cast<int32_t>(lane);
        if (at < n && ((rn[j].x >> kRecCntShift) & kRecCntMask) == 0u) hn[j] = p.hot[rn[j].y];
      }
      // ---- single-ELT events: uniform, table position, then both table reads, then the losses
      int mode[2];  // 0: none, 1: loss known (no loss / mean), 2: table, 3: Halley
      float val[2], sfrac[2];
      const float4* node[2];
      uint32_t lmask[2];  // the layers the event serves
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool valid = base + 32 * j + static_cast<int32_t>(lane) < n;
        const uint32_t cnt = ((r[j].x >> kRecCntShift) & kRecCntMask) + 1u;
        const uint32_t tl = kPerTrial ? tl0 : r[j].x >> kRecTrialShift;
        mode[j] = 0;
        val[j] = 0.0f;
        sfrac[j] = 0.0f;
        node[j] = nullptr;
        lmask[j] = (valid && cnt == 1u)
                       ? static_cast<uint32_t>(bs.layers_of[pair_pos(h[j].meta)]) & (kPerTrial ? act0 : ws.act[tl])
                       : 0u;
        if (lmask[j]) {
          const uint32_t kind = pair_kind(h[j].meta);
          const uint32_t pos = pair_pos(h[j].meta);
          mode[j] = 1;
          val[j] = h[j].mu;
          if (kind == kKindZero) {
            val[j] = 0.0f;
          } else if (!p.primary_only && kind_is_beta(kind)) {
            float t = 0.0f;
            if (p.newton_only || !pair_tab_exact(h[j].meta) ||
                !batch_pair_normal(p, kind, bs.elt_id[pos], r[j].y, ta + tl, r[j].x & kRecKMask, &t)) {
              mode[j] = 3;
            } else {
              mode[j] = 2;
              const bool fine = pair_fine(h[j].meta);
              const int nseg = fine ? kTabFineNodes - 1 : kTabNodes - 1;
              float u = (t + kTabT1f) * (fine ? kTabInvH * kTabRefine : kTabInvH);
              u = fminf(fmaxf(u, 0.0f), static_cast<float>(nseg));
              int i = static_cast<int>(u);
              if (i > nseg - 1) i = nseg - 1;
              sfrac[j] = u - static_cast<float>(i);
              node[j] = (fine ? bs.tabf[pos] : bs.tab[pos]) + h[j].node + i;
            }
          }
        }
      }
      float4 n0[2];
      float2 n1[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (mode[j] == 2) {
          n0[j] = __ldg(node[j]);
          n1[j] = __ldg(reinterpret_cast<const float2*>(node[j] + 1) + 1);
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (mode[j] == 0) continue;
        const uint32_t pos = pair_pos(h[j].meta);
        const uint32_t tl = kPerTrial ? tl0 : r[j].x >> kRecTrialShift;
        float L;
        if (mode[j] == 3) {
          L = pair_loss_slow(p, p.pairs[r[j].y], r[j].y, ta + tl, r[j].x & kRecKMask, &nc);
        } else {
          float loss = val[j];
          if (mode[j] == 2)
            loss = (n0[j].x > 0.0f)
                       ? h[j].max_l * (n0[j].x * expf(tab_increment(sfrac[j], n0[j].y, n0[j].z, n0[j].w, n1[j].x,
                                                                     n1[j].y)))
                       : 0.0f;
          L = bs.share[pos] * clamp_terms_f(loss, bs.ret[pos], bs.lim[pos]);
        }
        if constexpr (!kPerTrial) {
          if (tl != cur) {  // the lane's records have moved on to a later trial
            flush_lane(ws, lane, cur, dirty);
            dirty = 0u;
            cur = tl;
          }
        }
        for (uint32_t m = lmask[j]; m; m &= m - 1u) add_occurrence(ws, bs, __ffs(m) - 1, lane, L, &dirty);
        ++n_pairs;
      }
      // ---- multi-ELT events: queued
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool valid = base + 32 * j + static_cast<int32_t>(lane) < n;
        const bool multi = valid && ((r[j].x >> kRecCntShift) & kRecCntMask) != 0u;
        const uint32_t mmask = __ballot_sync(0xffffffffu, multi);
        if (mmask) {
          if (nq + __popc(mmask) > kBatchQueue) {
            __syncwarp();
            const uint32_t np = batch_multi<kPerTrial>(p, bs, ws, nq, ta, &nc);
            if (lane == 0) n_pairs += np;
            nq = 0;
          }
          if (multi) ws.mq[nq + __popc(mmask & lt_mask)] = r[j];
          nq += __popc(mmask);
          __syncwarp();
        }
      }
    }
    if (nq > 0) {
      const uint32_t np = batch_multi<kPerTrial>(p, bs, ws, nq, ta, &nc);
      if (lane == 0) n_pairs += np;
    }
    // ---- the year losses of the item's trials for each layer: the aggregate terms of the trials' sums
    if constexpr (kPerTrial) {
      __syncwarp();
      for (int l = static_cast<int>(lane); l < nl; l += 32) {  // the lanes' sums, one lane per layer
        unsigned long long S = 0ull;
        for (int j = 0; j < 32; ++j) S += ws.acc[l][j];
        const double sd = __ull2double_rn(S) * p.inv_scale[l];
        if (ta + t_lo < p.layer_t_end[l]) p.ylt_l[l][ta + t_lo - p.t_begin] = clamp_terms_d(sd, p.agg_r[l], p.agg_l[l]);
      }
    } else {
      flush_lane(ws, lane, cur, dirty);
      __syncwarp();
      for (int i = static_cast<int>(lane); i < nl * ntr; i += 32) {
        const int l = i / ntr, t = i - l * ntr;
        const double sd = __ull2double_rn(ws.tacc[l][t]) * p.inv_scale[l];
        if (ta + t < p.layer_t_end[l]) p.ylt_l[l][ta + t - p.t_begin] = clamp_terms_d(sd, p.agg_r[l], p.agg_l[l]);
      }
    }
    __syncwarp();
  }
  n_pairs = __reduce_add_sync(0xffffffffu, n_pairs);
  for (int d = 16; d > 0; d >>= 1) nc += __shfl_xor_sync(0xffffffffu, nc, d);
  if (lane == 0) {
    if (n_pairs) atomicAdd(&p.counters[1], static_cast<unsigned long long>(n_pairs));
    if (nc) atomicAdd(&p.counters[2], nc);
  }
}

namespace {

// ------------------------------------------------------------------ dense kernel
// One warp per tile, one lane per (event occurrence, ELT) pair.  The tile's
// records go by windows of up to 32 pairs of whole events.  Each pair's loss
// after ELT terms is computed once and stored with the layers it serves; then
// the lanes turn into layers: lane (s, l) holds layer l's fixed-point sum for
// the current trial in registers and takes the window's events i = s mod S (S
// event slots: 32 over the layers rounded up to a power of two) that serve
// layer l, found by a bit-matrix transpose of the events' layer masks.  For
// each (single-ELT events first, then the others), it sums the event's pair
// losses over the layer's ELTs from left to right (the pairs' order), applies
// the occurrence terms and adds the result.  When a trial's events are all
// taken, the slots' sums give its year losses.  An event of more than 32 pairs
// goes alone.
//
// Bound by issue (62% of the slots, ~730 instructions a window: the pairs'
// losses 200, the adds by layer 250, where a warp waits for its lane with the
// most events) and the conversions to fixed point.  16 layers over 64 ELTs,
// 150,001 trials of 320 pairs: 1,445 us (1,700 with records and pairs in rings,
// 64 pairs a round); 30,000 trials over a 100,000-event catalogue 1,480 (3,070).
// Two adds a step, or the conversion in integer arithmetic: the same or slower.
constexpr int kDenseBlocksPerSm = 7;  // 72 registers, 28 warps per SM (6: 1,520 us, 8: 1,550)

struct DenseWarp {
  float loss[kMaxIndexElts];      // a window's pair losses after ELT terms
  uint32_t lmask[kMaxIndexElts];  // and the pairs' layers: those holding its ELT that reach its trial
  float first[32];                // the window's events: the first pair's loss,
  uint32_t place[32];             //   the first pair and the pair count << 8
  uint32_t act[kWarpTrials];      // per trial of the tile: the layers whose trials reach it
};

struct DenseShared {
  const float4* tab[kMaxIndexElts];
  const float4* tabf[kMaxIndexElts];
  uint32_t elt_id[kMaxIndexElts];
  float ret[kMaxIndexElts], lim[kMaxIndexElts], share[kMaxIndexElts];
  uint32_t layers_of[kMaxIndexElts];
  float4 occ[kBatchLayers];  // (occurrence retention, occurrence limit, fixed-point scale, 0)
  double agg_r[kBatchLayers], agg_l[kBatchLayers], inv_scale[kBatchLayers];
  double* ylt[kBatchLayers];
  int64_t t_end[kBatchLayers];
};

// Loss after ELT terms by the Halley iteration, with its non-convergence as
// the second value (0 or 1).
__device__ __noinline__ float2 dense_pair_slow(const BatchParams& p, uint32_t pi, int64_t trial, uint32_t k) {
  unsigned long long nc = 0ull;
  const float L = pair_loss_slow(p, p.pairs[pi], pi, trial, k, &nc);
  return make_float2(L, static_cast<float>(nc));
}

// The pass's per-ELT and per-layer constants in shared memory (the caller syncs).
__device__ __forceinline__ void load_dense_shared(const BatchParams& p, DenseShared& ds) {
  const int nl = p.n_layers;
  for (int i = threadIdx.x; i < kMaxIndexElts; i += blockDim.x) {
    const bool in = i < p.n_elts;
    ds.tab[i] = in ? p.tab[i] : nullptr;
    ds.tabf[i] = in ? p.tabf[i] : nullptr;
    ds.elt_id[i] = in ? static_cast<uint32_t>(p.elt_id[i]) : 0u;
    ds.ret[i] = in ? p.t_ret[i] : 0.0f;
    ds.lim[i] = in ? p.t_lim[i] : 0.0f;
    ds.share[i] = in ? p.t_share[i] : 0.0f;
    ds.layers_of[i] = in ? static_cast<uint32_t>(p.layers_of[i]) : 0u;
  }
  for (int i = threadIdx.x; i < kBatchLayers; i += blockDim.x) {
    const bool in = i < nl;
    ds.occ[i] = make_float4(p.occ_r[i], p.occ_l[i], p.scale[i], 0.0f);
    ds.agg_r[i] = p.agg_r[i];
    ds.agg_l[i] = p.agg_l[i];
    ds.inv_scale[i] = p.inv_scale[i];
    ds.ylt[i] = in ? p.ylt_l[i] : nullptr;
    ds.t_end[i] = in ? p.layer_t_end[i] : 0;
  }
}

// Lane l receives column l of the 32 x 32 bit matrix whose row i is lane i's
// x: bit i of the result is bit l of lane i's x (the off-diagonal blocks of
// halves, quarters, ... exchanged between lanes).
__device__ __forceinline__ uint32_t bit_transpose32(uint32_t x, uint32_t lane) {
  const uint32_t hi[5] = {0xFFFF0000u, 0xFF00FF00u, 0xF0F0F0F0u, 0xCCCCCCCCu, 0xAAAAAAAAu};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const uint32_t j = 16u >> k;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & hi[k]) | ((y & hi[k]) >> j)) : ((x & ~hi[k]) | ((y & ~hi[k]) << j));
  }
  return x;
}

// Year losses of one trial: the slots' sums of each layer added (lanes l of
// slot 0 receive them) through the aggregate terms; the sums are cleared.
__device__ __forceinline__ void dense_finish_trial(const DenseShared& ds, unsigned long long& acc, uint32_t lane,
                                                   int nlp, int nl, int64_t trial, int64_t t_begin) {
  for (int d = nlp; d < 32; d <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
  if (lane < static_cast<uint32_t>(nl) && trial < ds.t_end[lane])
    ds.ylt[lane][trial - t_begin] =
        clamp_terms_d(__ull2double_rn(acc) * ds.inv_scale[lane], ds.agg_r[lane], ds.agg_l[lane]);
  acc = 0ull;
}

}  // namespace

namespace {

// A pair between its two halves: its loss known (a), from a table interval (a =
// max_l, s the place in the interval n0, n1), or by the Halley iteration.
struct DensePair {
  uint32_t layers;  // the pair's layers that reach its trial
  uint32_t mode, pos;
  float a, s;
  float4 n0;
  float2 n1;
};
enum : uint32_t { kDenseKnown = 0, kDenseTable = 1, kDenseSlow = 2 };

// The first half, for lanes with `in`: key is the record's first word, act the
// layers that reach its trial.
__device__ __forceinline__ DensePair dense_begin(const BatchParams& p, const DenseShared& ds, const DenseWarp& ws,
                                                 bool in, const PairHot& h, uint32_t pi, int64_t ta, uint32_t key) {
  DensePair e{0u, kDenseKnown, pair_pos(h.meta), 0.0f, 0.0f, make_float4(0.0f, 0.0f, 0.0f, 0.0f),
              make_float2(0.0f, 0.0f)};
  if (in) {
    const uint32_t tl = key >> kRecTrialShift;
    e.layers = ds.layers_of[e.pos] & ws.act[tl];
    if (e.layers) {
      const uint32_t kind = pair_kind(h.meta);
      e.a = kind == kKindZero ? 0.0f : h.mu;
      if (!p.primary_only && kind_is_beta(kind)) {
        float t;
        if (p.newton_only || !pair_tab_exact(h.meta) ||
            !batch_pair_normal(p, kind, ds.elt_id[e.pos], pi, ta + tl, key & kRecKMask, &t)) {
          e.mode = kDenseSlow;
        } else {
          const bool fine = pair_fine(h.meta);
          const TabPlace at = tab_place(t, fine);
          const float4* node = (fine ? ds.tabf[e.pos] : ds.tab[e.pos]) + h.node + at.i;
          e.mode = kDenseTable;
          e.a = h.max_l;
          e.s = at.s;
          e.n0 = __ldg(node);
          e.n1 = __ldg(reinterpret_cast<const float2*>(node + 1) + 1);
        }
      }
    }
  }
  return e;
}

// The second half: the pair's loss after ELT terms.
__device__ __forceinline__ float dense_end(const BatchParams& p, const DenseShared& ds, const DensePair& e,
                                           uint32_t pi, int64_t ta, uint32_t key, unsigned long long* nc) {
  if (e.mode == kDenseSlow) {
    const float2 r = dense_pair_slow(p, pi, ta + (key >> kRecTrialShift), key & kRecKMask);
    *nc += static_cast<unsigned long long>(r.y);
    return r.x;
  }
  float loss = e.a;
  if (e.mode == kDenseTable) loss = e.a * tab_value(e.s, e.n0, e.n1);
  return ds.share[e.pos] * clamp_terms_f(loss, ds.ret[e.pos], ds.lim[e.pos]);
}

// The sum, left to right, of the losses of pairs [first, first + n) that layer l holds.
__device__ __forceinline__ float dense_event_sum(const DenseWarp& ws, uint32_t first, uint32_t n, uint32_t l) {
  float G = 0.0f;
  for (uint32_t j = first; j < first + n; ++j)
    if ((ws.lmask[j] >> l) & 1u) G += ws.loss[j];
  return G;
}

// An event of more than 32 pairs, by the whole warp: its pairs' losses and layers into ws.
__device__ __noinline__ uint32_t dense_long_event(const BatchParams& p, const DenseShared& ds, DenseWarp& ws, uint2 r,
                                                  uint32_t cnt, int64_t ta, unsigned long long* nc) {
  uint32_t n_pairs = 0;
  for (uint32_t j = lane_id(); j < cnt; j += 32) {
    const uint32_t pi = r.y + j;
    const DensePair e = dense_begin(p, ds, ws, true, p.hot[pi], pi, ta, r.x);
    ws.loss[j] = dense_end(p, ds, e, pi, ta, r.x, nc);
    ws.lmask[j] = e.layers;
    n_pairs += e.layers != 0u;
  }
  __syncwarp();
  return n_pairs;
}

}  // namespace

__global__ void __launch_bounds__(kBatchThreads, kDenseBlocksPerSm)
    k_losses_dense(const __grid_constant__ BatchParams p) {
  __shared__ DenseWarp dwarp[kBatchThreads / 32];
  __shared__ DenseShared ds;
  const uint32_t lane = lane_id();
  DenseWarp& ws = dwarp[threadIdx.x >> 5];
  const int nl = p.n_layers;
  load_dense_shared(p, ds);
  __syncthreads();
  static_assert(kBatchLayers <= 32, "one lane per layer; 32-bit layer masks");
  // the lane's layer l and event slot s; its events in a window: i = s mod S
  int nlp = 1;
  while (nlp < nl) nlp <<= 1;
  const uint32_t my_l = lane & static_cast<uint32_t>(nlp - 1);
  const uint32_t n_slots = 32u / static_cast<uint32_t>(nlp);
  uint32_t my_pattern = 0u;
  for (uint32_t i = lane / static_cast<uint32_t>(nlp); i < 32u; i += n_slots) my_pattern |= 1u << i;
  if (my_l >= static_cast<uint32_t>(nl)) my_pattern = 0u;
  unsigned long long acc = 0ull;  // the layer's sum over the slot's events of the current trial
  unsigned long long nc = 0ull;
  uint32_t n_pairs = 0;

  unsigned long long next_tile = 0ull;  // tiles are claimed one ahead
  if (lane == 0) next_tile = atomicAdd(&p.counters[0], 1ull);
  for (;;) {
    const int64_t tile = static_cast<int64_t>(__shfl_sync(0xffffffffu, next_tile, 0));
    if (tile >= p.n_tiles) break;
    if (lane == 0) next_tile = atomicAdd(&p.counters[0], 1ull);
    const int64_t ta = p.t_begin + tile * p.tile_trials;
    const int ntr = static_cast<int>((ta + p.tile_trials < p.t_end) ? p.tile_trials : p.t_end - ta);
    uint32_t any = 0u;
#pragma unroll
    for (int t = 0; t < kWarpTrials; ++t) {
      const uint32_t a =
          __ballot_sync(0xffffffffu, t < ntr && lane < static_cast<uint32_t>(nl) && ta + t < ds.t_end[lane]);
      if (lane == 0) ws.act[t] = a;
      any |= a;
    }
    __syncwarp();
    const uint2* recs = p.ev_buf + (__ldg(&p.off[ta]) - p.e0);
    const uint32_t n = any ? __ldg(&p.tile_cnt[tile]) : 0u;
    // a window's table intervals are in flight while the next window is laid out, that one's hot records
    // while this one's sums are made, and the records after it meanwhile
    auto count_of = [](uint2 x) { return ((x.x >> kRecCntShift) & kRecCntMask) + 1u; };
    uint2 r = lane < n ? __ldg(recs + lane) : make_uint2(0u, 0u);
    uint32_t next = 0u;  // the first record after the window
    PairWindow w;
    PairHot h;
    uint32_t evx;  // of lane i < n_take: the window's event i's record's first word
    auto next_window = [&]() {
      w = make_window(r, next + lane < n ? count_of(r) : 0u);
      evx = r.x;
      h = PairHot{0.0f, 0.0f, kKindZero << kMetaKindShift, 0u};
      if (lane < w.np) h = p.hot[w.ey + (lane - w.epre)];
      if (w.n_take > 0) {
        next += static_cast<uint32_t>(w.n_take);
        if (next + lane < n) r = __ldg(recs + next + lane);
      }
    };
    next_window();
    int cur = 0;  // the trial whose events are being taken
    for (;;) {
      if (w.np == 0u) {
        if (next >= n) break;
        // the next event has more than 32 pairs
        const uint2 x = make_uint2(__shfl_sync(0xffffffffu, r.x, 0), __shfl_sync(0xffffffffu, r.y, 0));
        for (; cur < static_cast<int>(x.x >> kRecTrialShift); ++cur)
          dense_finish_trial(ds, acc, lane, nlp, nl, ta + cur, p.t_begin);
        const uint32_t cnt = count_of(x);
        n_pairs += dense_long_event(p, ds, ws, x, cnt, ta, &nc);
        if (lane < static_cast<uint32_t>(nl)) {
          const float4 oc = ds.occ[lane];
          acc += fixed_units(clamp_terms_f(dense_event_sum(ws, 0u, cnt, lane), oc.x, oc.y), oc.z);
        }
        __syncwarp();
        ++next;
        if (next + lane < n) r = __ldg(recs + next + lane);
        next_window();
        continue;
      }
      const uint32_t pi = w.ey + (lane - w.epre), key = w.ex, np = w.np;
      const DensePair e = dense_begin(p, ds, ws, lane < np, h, pi, ta, key);
      const uint32_t n_take = static_cast<uint32_t>(w.n_take), ev_first = w.pre, ev_key = evx;
      next_window();
      ws.loss[lane] = dense_end(p, ds, e, pi, ta, key, &nc);
      ws.lmask[lane] = e.layers;
      n_pairs += e.layers != 0u;
      __syncwarp();
      // lane i as event i: the layers it serves
      uint32_t m = 0u, cnt = 0u;
      int t = -1;
      if (lane < n_take) {
        cnt = ((ev_key >> kRecCntShift) & kRecCntMask) + 1u;
        t = static_cast<int>(ev_key >> kRecTrialShift);
        m = ws.lmask[ev_first];
        for (uint32_t j = 1; j < cnt; ++j) m |= ws.lmask[ev_first + j];
        ws.first[lane] = ws.loss[ev_first];
        ws.place[lane] = ev_first | cnt << 8;
      }
      const uint32_t multi = __ballot_sync(0xffffffffu, cnt > 1u);
      // lane (s, l): the slot's events that serve layer l
      const uint32_t col = __shfl_sync(0xffffffffu, bit_transpose32(m, lane), my_l) & my_pattern;
      __syncwarp();
      const float4 oc = ds.occ[my_l];  // the layer's occurrence terms and fixed-point scale
      for (uint32_t done = 0; done < n_take;) {  // by trial
        const int tr = __shfl_sync(0xffffffffu, t, done);
        for (; cur < tr; ++cur) dense_finish_trial(ds, acc, lane, nlp, nl, ta + cur, p.t_begin);
        // (records are in trial order; <= keeps the loop finite whatever the order)
        const uint32_t seg = __ballot_sync(0xffffffffu, lane >= done && lane < n_take && t <= tr);
        for (uint32_t one = col & seg & ~multi; one;) {  // events of one pair
          const int i = 31 - __clz(one);
          one ^= 1u << i;
          acc += fixed_units(clamp_terms_f(ws.first[i], oc.x, oc.y), oc.z);
        }
        for (uint32_t many = col & seg & multi; many;) {
          const int i = 31 - __clz(many);
          many ^= 1u << i;
          const uint32_t pl = ws.place[i];
          acc += fixed_units(clamp_terms_f(dense_event_sum(ws, pl & 0xffu, pl >> 8, my_l), oc.x, oc.y), oc.z);
        }
        done += __popc(seg);
      }
      __syncwarp();  // the window's losses are rewritten
    }
    for (; cur < ntr; ++cur) dense_finish_trial(ds, acc, lane, nlp, nl, ta + cur, p.t_begin);
    __syncwarp();
  }
  n_pairs = __reduce_add_sync(0xffffffffu, n_pairs);
  for (int d = 16; d > 0; d >>= 1) nc += __shfl_xor_sync(0xffffffffu, nc, d);
  if (lane == 0) {
    if (n_pairs) atomicAdd(&p.counters[1], static_cast<unsigned long long>(n_pairs));
    if (nc) atomicAdd(&p.counters[2], nc);
  }
}

int losses_dense_blocks_per_sm(int /*n_layers*/) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_losses_dense, kBatchThreads, 0) != cudaSuccess) return 0;
  return b;
}

cudaError_t launch_losses_batch(const BatchParams& p, int item, int grid, cudaStream_t s) {
  switch (item) {
    case kItemTile:
      k_losses_batch<false><<<grid, kBatchThreads, 0, s>>>(p);
      break;
    case kItemTrial:
      k_losses_batch<true><<<grid, kBatchThreads, 0, s>>>(p);
      break;
    case kItemDense:
      k_losses_dense<<<grid, kBatchThreads, 0, s>>>(p);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}


// ------------------------------------------------------------------ indexed kernel
// A warp per distinct event of the pass's ELT union and trial slice (claimed
// from the slice's queue, eight events at a time), over the event's
// occurrences in the slice, 32 at a time (a lane each).  The slice's bounds
// come from the index's trial grid, with a warp search only where a bound is
// inside a grid cell (a pass's ends off the grid).  Every lane of
// the warp works on the same event, so the pairs, their layers and their
// tables are the same across the warp.  For each occurrence and each layer it
// serves, the event's pair losses over the layer's ELTs are summed from left
// to right (per-lane running sums in shared memory when the event has several
// pairs), the occurrence terms applied, and the result added to the trial's
// fixed-point sum with a 64-bit atomic add: the same numbers as the other
// work items, so the same bits.  A second kernel turns the sums into year
// losses.
//
// Cost: issue (70% of the slots; Philox, Phi^-1 and the table are most of the
// ~350 instructions a window of 32 occurrences) and, before, the adds: L2 takes
// 8-byte adds to scattered sectors at 210 G/s at most, two in a sector at 360,
// four at 450.  So a trial's sums stand side by side, and the adds of a window
// go by lanes of four with three or more layers (a lane a layer).  Events of
// one pair with an exact table, nearly all, keep the pair's fields in registers
// over their windows, and the next window is loaded ahead.  16 layers over 64
// ELTs, 1M trials of 1,000 events: 4,200 us, 5,195 with an add per layer from
// each occurrence's lane, sums by layer and the fields loaded per window.
// 32 warps an SM (64 registers, a few spilled outside the window) against 28:
// 4,200 and 4,330 us; 36: 4,315.
namespace {

constexpr int kIdxThreads = 128;
constexpr int kIdxBlocksPerSm = 8;
constexpr int kIdxClaim = 8;  // events a warp claims at a time

struct IdxWarp {
  uint32_t pmask[kMaxIndexElts];     // the event's pairs: layers holding their ELTs
  float4 held[32];                   // the layers that the event serves, ascending: occurrence terms, scale, byte offset
                                     // in a trial's sums
  uint32_t last[32];                 // ... their last trials
  uint32_t trial[32];                // a window's trials
  uint32_t lay[32];                  // ... and their numbers
  uint4 meta[2 * kIdxClaim];         // the claimed events: [j] (first pair, pair end, range of the slice's first
                                     // occurrence), [kIdxClaim + j] (range of its end, -, -)
  int64_t span[2];                   // the trials of the claim's slice
};

// First entry in [lo, hi) of the event's occurrences whose trial is >= key
// (hi if none), by the whole warp: each round probes 32 evenly spaced entries.
// (An index holds up to 2^32 - 2 occurrences: probes past hi are in 64 bits.)
__device__ __forceinline__ uint32_t first_occ_at(const unsigned long long* occ, uint32_t lo, uint32_t hi,
                                                 int64_t key, uint32_t lane) {
  while (lo < hi) {
    const uint32_t step = (hi - lo - 1u) / 32u + 1u;
    const uint64_t pos = static_cast<uint64_t>(lo) + lane * step;
    const bool ge = pos < hi && static_cast<int64_t>(__ldg(occ + pos) >> 32) >= key;
    const uint32_t b = __ballot_sync(0xffffffffu, ge);
    if (b == 0u) {
      const uint32_t probes = (hi - lo - 1u) / step + 1u;
      lo += (probes - 1u) * step + 1u;
    } else {
      const uint32_t f = static_cast<uint32_t>(__ffs(b) - 1);
      hi = lo + f * step;
      if (f > 0u) lo += (f - 1u) * step + 1u;
    }
  }
  return lo;
}

// Loss after ELT terms of pair pi in occurrence (trial, k): as the other work items compute it.
__device__ __forceinline__ float indexed_pair_loss(const BatchParams& p, const DenseShared& ds, uint32_t pi,
                                                   int64_t trial, uint32_t k, unsigned long long* nc) {
  const PairHot h = p.hot[pi];
  const uint32_t kind = pair_kind(h.meta);
  const uint32_t pos = pair_pos(h.meta);
  float loss = h.mu;
  if (kind == kKindZero) {
    loss = 0.0f;
  } else if (!p.primary_only && kind_is_beta(kind)) {
    float t;
    if (p.newton_only || !pair_tab_exact(h.meta) || !batch_pair_normal(p, kind, ds.elt_id[pos], pi, trial, k, &t))
      return pair_loss_slow(p, p.pairs[pi], pi, trial, k, nc);
    const bool fine = pair_fine(h.meta);
    loss = h.max_l * tab_quantile_t((fine ? ds.tabf[pos] : ds.tab[pos]) + h.node, t, fine);
  }
  return ds.share[pos] * clamp_terms_f(loss, ds.ret[pos], ds.lim[pos]);
}

}  // namespace

__global__ void __launch_bounds__(kIdxThreads, kIdxBlocksPerSm)
    k_losses_indexed(const __grid_constant__ IndexedParams q) {
  const BatchParams& p = q.b;
  __shared__ IdxWarp iwarp[kIdxThreads / 32];
  __shared__ DenseShared ds;
  const uint32_t lane = lane_id();
  IdxWarp& ws = iwarp[threadIdx.x >> 5];
  // per warp, layer and lane: the running sum of an occurrence's pair losses (of events of several pairs)
  extern __shared__ float4 idx_gacc[];
  float (*gacc)[32] = reinterpret_cast<float (*)[32]>(idx_gacc) + (threadIdx.x >> 5) * p.n_layers;
  load_dense_shared(p, ds);
  __syncthreads();
  const int nl = p.n_layers;
  const int64_t t0 = p.t_begin;
  int64_t t_full = p.t_end;  // below it every layer reaches the trial
  for (int l = 0; l < nl; ++l) t_full = min(t_full, ds.t_end[l]);
  const uint32_t all = nl >= 32 ? 0xffffffffu : (1u << nl) - 1u;
  for (int l = 0; l < nl; ++l) gacc[l][lane] = 0.0f;
  const uint32_t n_u = *q.n_u;
  const uint32_t row_bytes = 8u * static_cast<uint32_t>(nl);
  char* const acc0 = reinterpret_cast<char*>(q.acc - t0 * nl);
  unsigned long long nc = 0ull;
  uint32_t n_pairs = 0;
  // the occurrences (read once) are the first to leave L2, so that the trials' sums, which the atomic
  // adds revisit, stay (batched-16: 5.98 against 6.07 ms a pass)
  uint64_t occ_pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(occ_pol));

  auto load_occ = [&](const unsigned long long* at) {
    unsigned long long o;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u64 %0, [%1], %2;" : "=l"(o) : "l"(at), "l"(occ_pol));
    return o;
  };

  // the queue's groups: kIdxClaim events over one trial slice, every event of a slice before the next
  // slice, so that the sums being added to stay within a slice's trials; a warp moves to the next slice
  // when the slice's queue runs out. For the group's event j, lane j loads its pairs and the grid range
  // that holds the slice's first occurrence, lane kIdxClaim + j the range that holds the slice's end (a
  // bound on the grid is its own range); the next group's loads are issued before this group's events run.
  const int slice_shift = q.slice_shift, grid_shift = q.grid_shift;
  const int64_t k0 = t0 >> slice_shift;
  const uint32_t per_slice = (n_u + kIdxClaim - 1) / kIdxClaim;
  const uint32_t n_slices = static_cast<uint32_t>(indexed_slices(t0, p.t_end, slice_shift));
  uint4 meta = make_uint4(0u, 0u, 0u, 0u);
  uint32_t sl = 0u;  // the slice of the group claimed last
  auto slice_lo = [&](uint32_t j) { return max(t0, (k0 + j) << slice_shift); };
  auto slice_hi = [&](uint32_t j) { return min(p.t_end, (k0 + j + 1) << slice_shift); };
  auto claim = [&]() {
    uint32_t g = 0u;
    for (; sl < n_slices; ++sl) {
      if (lane == 0) g = atomicAdd(q.slice_queue + sl, 1u);
      g = __shfl_sync(0xffffffffu, g, 0);
      if (g < per_slice) break;
    }
    const uint32_t j = lane & static_cast<uint32_t>(kIdxClaim - 1), u = g * kIdxClaim + j;
    if (sl < n_slices && lane < static_cast<uint32_t>(2 * kIdxClaim) && u < n_u) {
      const uint32_t* row = q.ev_grid + static_cast<int64_t>(q.u_event[u]) * (q.grid_cells + 1);
      const bool end = lane >= static_cast<uint32_t>(kIdxClaim);
      const int64_t b = end ? slice_hi(sl) : slice_lo(sl);
      const int64_t cell = b >= q.yet_trials ? q.grid_cells : b >> grid_shift;
      const bool on_grid = b >= q.yet_trials || (b & ((int64_t{1} << grid_shift) - 1)) == 0;
      const uint32_t x = row[cell], y = on_grid ? x : row[cell + 1];
      meta = end ? make_uint4(x, y, 0u, 0u) : make_uint4(q.u_first[u], q.u_first[u + 1], x, y);
    }
    return g;
  };
  uint32_t grp = claim();
  while (sl < n_slices) {
    if (lane < static_cast<uint32_t>(2 * kIdxClaim)) ws.meta[lane] = meta;
    if (lane == 0) {
      ws.span[0] = slice_lo(sl);
      ws.span[1] = slice_hi(sl);
    }
    __syncwarp();
    const int n_here = static_cast<int>(min(static_cast<uint32_t>(kIdxClaim), n_u - grp * kIdxClaim));
    grp = claim();
    for (int g = 0; g < n_here; ++g) {
      const uint4 m4 = ws.meta[g], h4 = ws.meta[kIdxClaim + g];
      const uint32_t ps = m4.x, cnt = m4.y - m4.x;
      // the slice's occurrences: a search only where a bound is inside a grid cell
      const uint32_t lo = first_occ_at(q.occ, m4.z, m4.w, ws.span[0], lane);
      const uint32_t hi = first_occ_at(q.occ, max(lo, h4.x), h4.y, ws.span[1], lane);
      if (lo >= hi) continue;
      uint32_t touched = 0u;  // the event's layers
      for (uint32_t j = lane; j < cnt; j += 32) {
        const uint32_t m = ds.layers_of[pair_pos(p.hot[ps + j].meta)];
        ws.pmask[j] = m;
        touched |= m;
      }
      touched = __reduce_or_sync(0xffffffffu, touched);
      const int n_held = __popc(touched);
      if ((touched >> lane) & 1u) {
        const int at = __popc(touched & ((1u << lane) - 1u));
        const float4 oc = ds.occ[lane];
        ws.held[at] = make_float4(oc.x, oc.y, oc.z, __uint_as_float(8u * lane));
        ws.lay[at] = lane;
        ws.last[at] = static_cast<uint32_t>(ds.t_end[lane] - 1);
      }
      __syncwarp();
      unsigned long long o_next = 0ull;
      if (lane < hi - lo) o_next = load_occ(q.occ + lo + lane);
      auto layers_at = [&](uint32_t trial) {  // the layers whose trials reach this one
        uint32_t act = all;
        if (trial >= t_full) {
          act = 0u;
          for (int l = 0; l < nl; ++l)
            if (trial < ds.t_end[l]) act |= 1u << l;
        }
        return act;
      };
      auto add = [&](uint32_t tj, float G, const float4& h, uint32_t last, bool on) {
        const float O = clamp_terms_f(G, h.x, h.y);
        if (on && tj <= last && O > 0.0f)
          atomicAdd(reinterpret_cast<unsigned long long*>(acc0 + (static_cast<uint64_t>(tj) * row_bytes +
                                                                  __float_as_uint(h.w))),
                    fixed_units(O, h.z));
      };
      const PairHot h0 = p.hot[ps];
      const uint32_t kind = pair_kind(h0.meta), pos = pair_pos(h0.meta);
      if (cnt == 1u && kind_is_beta(kind) && pair_tab_exact(h0.meta) && !p.primary_only && !p.newton_only) {
        // most events: one pair, its loss from a table; the pair's fields stay in registers over the event
        const bool fine = pair_fine(h0.meta);
        const float4* const tab = (fine ? ds.tabf[pos] : ds.tab[pos]) + h0.node;
        const uint32_t elt = ds.elt_id[pos];
        const float ret = ds.ret[pos], lim = ds.lim[pos], share = ds.share[pos];
        for (uint32_t r = lo;; r += 32) {  // (windows by what is left: r + 32 may lie beyond 32 bits)
          const uint32_t left = hi - r;
          const unsigned long long o = o_next;
          if (lane + 32u < left) o_next = load_occ(q.occ + (r + lane + 32u));
          uint32_t trial = 0xffffffffu;  // above every layer's last trial
          float L = 0.0f;
          if (lane < left) {
            trial = static_cast<uint32_t>(o >> 32);
            if (touched & layers_at(trial)) {
              ++n_pairs;
              float t;
              if (batch_pair_normal(p, kind, elt, ps, trial, static_cast<uint32_t>(o), &t))
                L = share * clamp_terms_f(h0.max_l * tab_quantile_t(tab, t, fine), ret, lim);
              else
                L = pair_loss_slow(p, p.pairs[ps], ps, trial, static_cast<uint32_t>(o), &nc);
            }
          }
          // the adds: three or four layers at a time go by lanes of four (lane c of four adds the c-th layer of the
          // four's occurrences in turn, so that a trial's adds to one sector leave together), two by lanes of two,
          // one by each occurrence's own lane
          int at = 0;
          if (n_held >= 3) {
            uint32_t tq[4];
            float Lq[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              tq[c] = __shfl_sync(0xffffffffu, trial, (lane & 28u) + c);
              Lq[c] = __shfl_sync(0xffffffffu, L, (lane & 28u) + c);
            }
            for (; n_held - at >= 3; at += 4) {
              const int slot = at + static_cast<int>(lane & 3u);  // at most 31
              const float4 h = ws.held[slot];
              const uint32_t last = ws.last[slot];
#pragma unroll
              for (int c = 0; c < 4; ++c) add(tq[c], Lq[c], h, last, slot < n_held);
            }
          }
          if (n_held - at == 2) {
            const float4 h = ws.held[at + (lane & 1u)];
            const uint32_t last = ws.last[at + (lane & 1u)];
            for (uint32_t c = 0; c < 2; ++c) {
              const uint32_t src = (lane & 30u) + c;
              const uint32_t tj = __shfl_sync(0xffffffffu, trial, src);
              add(tj, __shfl_sync(0xffffffffu, L, src), h, last, true);
            }
          } else if (n_held - at == 1) {
            add(trial, L, ws.held[at], ws.last[at], true);
          }
          if (left <= 32u) break;
        }
      } else {
        for (uint32_t r = lo;; r += 32) {  // (windows by what is left: r + 32 may lie beyond 32 bits)
          const uint32_t left = hi - r;
          const unsigned long long o = o_next;
          if (lane + 32u < left) o_next = load_occ(q.occ + (r + lane + 32u));
          const uint32_t trial = static_cast<uint32_t>(o >> 32);
          const uint32_t act = lane < left ? layers_at(trial) : 0u;
          // the pairs in order: each layer's running sum is the left-to-right sum of its pairs' losses
          for (uint32_t j = 0; j < cnt; ++j) {
            const uint32_t m = ws.pmask[j] & act;
            if (m) {
              const float L = indexed_pair_loss(p, ds, ps + j, trial, static_cast<uint32_t>(o), &nc);
              ++n_pairs;
              for (uint32_t mm = m; mm; mm &= mm - 1u) gacc[__ffs(mm) - 1][lane] += L;
            }
          }
          ws.trial[lane] = lane < left ? trial : 0xffffffffu;
          __syncwarp();
          // the adds, by lanes of four as above
          for (int at = 0; at < n_held; at += 4) {
            const int slot = at + static_cast<int>(lane & 3u);
            if (slot >= n_held) continue;
            const float4 h = ws.held[slot];
            const uint32_t last = ws.last[slot];
            const float4 G = *reinterpret_cast<const float4*>(&gacc[ws.lay[slot]][lane & 28u]);
            const float Gq[4] = {G.x, G.y, G.z, G.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
              add(ws.trial[(lane & 28u) + c], Gq[c], h, last, true);
          }
          __syncwarp();
          for (uint32_t mm = touched; mm; mm &= mm - 1u) gacc[__ffs(mm) - 1][lane] = 0.0f;
          if (left <= 32u) break;
        }
      }
      __syncwarp();  // pmask is rewritten for the next event
    }
    __syncwarp();  // meta is rewritten for the next claim
  }
  n_pairs = __reduce_add_sync(0xffffffffu, n_pairs);
  for (int d = 16; d > 0; d >>= 1) nc += __shfl_xor_sync(0xffffffffu, nc, d);
  if (lane == 0) {
    if (n_pairs) atomicAdd(&p.counters[1], static_cast<unsigned long long>(n_pairs));
    if (nc) atomicAdd(&p.counters[2], nc);
  }
}

namespace {

// The year loss of a fixed-point sum: clamp_terms_d(sum * inv_scale, r, l) with
// FP64 instructions for the conversion and the subtraction only (the FP64 pipe
// bound the kernel below: 1M trials of 16 layers 79 us, 128 with all of it in
// FP64): inv_scale is a power of two whose product with a
// sum is normal, so it adds to the exponent, and doubles that are not negative
// are ordered as their bits.
__device__ __forceinline__ double year_loss(unsigned long long sum, double inv_scale, double r, double l) {
  const long long x = __double_as_longlong(__ull2double_rn(sum)) + __double_as_longlong(inv_scale) -
                      __double_as_longlong(1.0);
  long long d = __double_as_longlong(__longlong_as_double(sum ? x : 0ll) - r);
  d = d < 0ll ? 0ll : d;
  const long long lim = __double_as_longlong(l);
  return __longlong_as_double(d < lim ? d : lim);
}

__global__ void k_indexed_years(const __grid_constant__ IndexedParams q) {
  const BatchParams& p = q.b;
  const int64_t n = p.t_end - p.t_begin;
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t tt = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; tt < n; tt += step)
    for (int l = 0; l < p.n_layers; ++l)
      if (p.t_begin + tt < p.layer_t_end[l])
        p.ylt_l[l][tt] = year_loss(q.acc[tt * p.n_layers + l], p.inv_scale[l], p.agg_r[l], p.agg_l[l]);
}

size_t idx_smem_bytes(int n_layers) { return sizeof(float) * kIdxThreads * n_layers; }

int grid_for_n(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return static_cast<int>(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

}  // namespace

int losses_indexed_blocks_per_sm(int n_layers) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_losses_indexed, kIdxThreads, idx_smem_bytes(n_layers)) != cudaSuccess) return 0;
  return b;
}

cudaError_t launch_losses_indexed(const IndexedParams& q, int grid, cudaStream_t s) {
  k_losses_indexed<<<grid, kIdxThreads, idx_smem_bytes(q.b.n_layers), s>>>(q);
  return cudaGetLastError();
}

cudaError_t launch_indexed_years(const IndexedParams& q, cudaStream_t s) {
  k_indexed_years<<<grid_for_n(q.b.t_end - q.b.t_begin, 256), 256, 0, s>>>(q);
  return cudaGetLastError();
}


}  // namespace ara
