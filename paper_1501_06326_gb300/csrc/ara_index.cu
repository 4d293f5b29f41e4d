// Event-major index of a resident YET: for each catalogue event, its
// occurrences (trial, event index in the trial), in trial order.  Built once
// per YET (ara_build_yet_index); batched passes then reach a layer's hit
// events through its ELTs' events instead of streaming every trial's events
// (Section 2.1's lookup, taken from the ELT side).
#include <cuda_runtime.h>

#include <cstdint>

#include "ara_batch.h"

namespace ara {

namespace {

// key = event id, value = (trial << 32) | event index: one warp per trial
__global__ void k_yet_pairs(const int64_t* __restrict__ off, const int32_t* __restrict__ ids, int64_t n_trials,
                            unsigned long long* keys, int64_t* vals) {
  const uint32_t lane = threadIdx.x & 31u;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5); t < n_trials;
       t += warps) {
    const int64_t a = off[t], b = off[t + 1];
    for (int64_t i = a + lane; i < b; i += 32) {
      keys[i] = static_cast<unsigned long long>(static_cast<uint32_t>(ids[i]));
      vals[i] = (t << 32) | (i - a);
    }
  }
}

__global__ void k_fill_u32(uint32_t* a, int64_t n, uint32_t v) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) a[i] = v;
}

// ev_off[e] = the first sorted position of event e (an event without
// occurrences takes the next event's start; events past the last key keep n)
__global__ void k_event_starts(const unsigned long long* __restrict__ keys, int64_t n, uint32_t* ev_off) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    const int64_t cur = static_cast<int64_t>(keys[i]);
    const int64_t prev = i > 0 ? static_cast<int64_t>(keys[i - 1]) : -1;
    for (int64_t e = prev + 1; e <= cur; ++e) ev_off[e] = static_cast<uint32_t>(i);
  }
}

// ev_grid[e * (cells + 1) + k] = the first of event e's occurrences with
// trial >= k << grid_shift, by binary search within e's range
__global__ void k_event_grid(const unsigned long long* __restrict__ occ, const uint32_t* __restrict__ ev_off,
                             int64_t n_entries, int64_t cells, int grid_shift, uint32_t* ev_grid) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n_entries; i += stride) {
    const int64_t e = i / (cells + 1), k = i - e * (cells + 1);
    const int64_t key = k << grid_shift;
    uint32_t lo = ev_off[e], hi = ev_off[e + 1];
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2u;
      if (static_cast<int64_t>(occ[mid] >> 32) < key) lo = mid + 1u;
      else hi = mid;
    }
    ev_grid[i] = lo;
  }
}

// ---- the bucket build: occurrences counted, placed and sorted per (event, grid cell)

// cnt[e * cells1 + (t >> grid_shift)] += 1 for each event e of trial t: a warp per trial
__global__ void k_count_cells(const int64_t* __restrict__ off, const int32_t* __restrict__ ids, int64_t n_trials,
                              int64_t cells1, int grid_shift, uint32_t* cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5); t < n_trials;
       t += warps) {
    const int64_t a = off[t], b = off[t + 1], c = t >> grid_shift;
    for (int64_t i = a + lane; i < b; i += 32)
      atomicAdd(cnt + static_cast<int64_t>(ids[i]) * cells1 + c, 1u);
  }
}

__global__ void k_max_u32(const uint32_t* __restrict__ a, int64_t n, uint32_t* out) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  uint32_t m = 0u;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) m = max(m, a[i]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31u) == 0u && m) atomicMax(out, m);
}

// Each occurrence of an event in [e_lo, e_hi) to a slot of its (event, cell)
// bucket, claimed with an atomic add (the order within a bucket is the claims'
// order, then sorted).  The trials go in order, so each event of the range has
// one partly written line at a time; a range of 2^18 events keeps fewer of them
// in L2 at once (paper-1m: 39 ms a build against 42 ms at 2^19 events, 51 ms at
// 2^20, 84 ms in one pass, 49 ms at 2^17 with its 16 reads of the ids).
__global__ void k_scatter_cells(const int64_t* __restrict__ off, const int32_t* __restrict__ ids, int64_t n_trials,
                                int64_t cells1, int grid_shift, int32_t e_lo, int32_t e_hi,
                                const uint32_t* __restrict__ ev_grid, uint32_t* __restrict__ cur,
                                unsigned long long* __restrict__ occ) {
  constexpr int kU = 8;  // a lane's claims in flight before its stores
  const uint32_t lane = threadIdx.x & 31u;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5); t < n_trials;
       t += warps) {
    const int64_t a = off[t], b = off[t + 1], c = t >> grid_shift;
    for (int64_t i0 = a + lane; i0 < b; i0 += 32 * kU) {
      int64_t cell[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int64_t i = i0 + 32 * u;
        const int32_t e = i < b ? ids[i] : -1;
        cell[u] = (e >= e_lo && e < e_hi) ? static_cast<int64_t>(e) * cells1 + c : -1;
      }
      uint32_t slot[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (cell[u] >= 0) slot[u] = ev_grid[cell[u]] + atomicAdd(cur + cell[u], 1u);
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (cell[u] >= 0)
          occ[slot[u]] = (static_cast<unsigned long long>(t) << 32) | static_cast<unsigned long long>(i0 + 32 * u - a);
    }
  }
}

// Each bucket in ascending (trial, event index) order: a thread per bucket, an
// insertion sort (the claims come nearly in trial order, as the warps take the
// trials in order, so few elements move)
__global__ void k_sort_cells(const uint32_t* __restrict__ ev_grid, int64_t n_buckets, unsigned long long* occ) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t bk = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; bk < n_buckets; bk += stride) {
    const uint32_t lo = ev_grid[bk], hi = ev_grid[bk + 1];
    if (hi - lo < 2u) continue;
    unsigned long long prev = occ[lo];
    for (uint32_t i = lo + 1u; i < hi; ++i) {
      const unsigned long long v = occ[i];
      if (v >= prev) {
        prev = v;
        continue;
      }
      uint32_t j = i;  // v goes below position i: shift the larger ones up
      do {
        occ[j] = occ[j - 1u];
        --j;
      } while (j > lo && occ[j - 1u] > v);
      occ[j] = v;
    }
  }
}

// ---- the partition build: two stable partitions by event id, staged in shared memory
//
// The first partition places the occurrences by the id's high digit, packed as
// (low digit << 53 | trial << 22 | event index), into a buffer of 8 bytes an
// event; the second partitions each of those buckets by the low digit and
// unpacks.  Both keep the (trial, event index) order, so no sort follows.
// It moves 4 B an event for the first count, 4 + 8 for the first partition, 8
// for the second count, 8 + 8 for the second partition.
// Stores go out in runs of one digit (about 8 occurrences, 64 bytes, of a tile
// of 16,384 at 2,048 digits), where the bucket build's atomic slot claims store
// 8 bytes at a time; tiles follow one another in a segment, so the next run of
// a digit completes the line in L2.  Each partition of 400M occurrences takes
// about 2.7 ms (its counts 0.26 and 0.46 ms at the copy's rate), bound by shared
// memory and its latency at 16 warps an SM: issue 31%.  One CTA of 512 threads
// an SM with the next tile's items loaded while a tile goes out; without that
// 3.6 ms, and as two CTAs of 256 threads with tiles of 8,192 (runs half as long)
// 3.5 ms.  The build: 6.4 ms at 400,000 trials x 1,000 events, against 14.9 ms
// by buckets.

constexpr int kPartThreads = 512;
constexpr int kPartWarps = kPartThreads / 32;
constexpr int kPartItems = 32;                          // occurrences a lane holds
constexpr int kPartTile = kPartThreads * kPartItems;    // 16,384: 128 KB of staging
constexpr int kPartDigits = 2048;                       // digits of a partition, at most
constexpr int kPartKBits = 22, kPartTrialBits = 31;     // event index, trial (64 = 11 + 31 + 22)
constexpr uint32_t kPartNone = 0xFFFFu;                 // no occurrence in this slot
constexpr uint32_t kPartCntBits = 11;                   // a warp's count of a digit (at most 1,024), then a lane
constexpr uint32_t kPartCntMask = (1u << kPartCntBits) - 1u;
static_assert(32 * kPartItems <= 1024 && kPartDigits % (2 * kPartThreads) == 0, "counts fit, digits split evenly");

struct PartShared {
  unsigned long long stage[kPartTile];
  union {
    uint16_t wc[kPartWarps][kPartDigits];  // per warp: a digit's count, then the first place of its items
    uint16_t dig[kPartTile];               // the staged items' digits
  };
  uint32_t run[kPartDigits];  // the segment's next output position of each digit
  uint32_t gb[kPartDigits];   // output position - place in the tile
  uint32_t wsum[kPartWarps];
};

// The trial of YET position pos for a whole warp: the last t with off[t] <= pos
// < off[t + 1], from a t known to be at or below it.  32 probes a round, their
// spacing growing until one is past pos, then closing in.
__device__ __forceinline__ int64_t warp_trial_of(const int64_t* __restrict__ off, int64_t n_trials, int64_t t,
                                                 int64_t pos, uint32_t lane) {
  int64_t step = 1;
  for (;;) {
    const int64_t q = t + 1 + static_cast<int64_t>(lane) * step;
    const bool past = q >= n_trials || __ldg(off + q) > pos;
    const uint32_t b = __ballot_sync(0xffffffffu, past);
    const int first = b ? __ffs(b) - 1 : 32;  // probes before it are at or below pos
    if (first > 0) t += 1 + static_cast<int64_t>(first - 1) * step;
    if (b == 0u) step *= 32;
    else if (step == 1) return t;
    else step = step > 32 ? step / 32 : 1;
  }
}

// Partitions items [begin, end) in tiles of kPartTile by digit, each digit's
// items in order from sm.run[digit] on.  kFirst: the items are YET positions
// (ids, off), packed into out; else they are first-partition items (in),
// unpacked into out.
template <bool kFirst>
__device__ __forceinline__ void partition_items(PartShared& sm, const int64_t* __restrict__ off,
                                                const int32_t* __restrict__ ids, int64_t n_trials, int lo_bits,
                                                const unsigned long long* __restrict__ in, int64_t begin, int64_t end,
                                                int n_digits, unsigned long long* __restrict__ out) {
  n_digits = (n_digits + 7) & ~7;  // whole 16-byte words; the digits past the last have no items
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const int w0 = static_cast<int>(warp) * 32 * kPartItems;  // the warp's items of a tile: w0 + 32 j + lane
  int64_t tw = 0;  // kFirst: a trial at or below the warp's items
  unsigned long long v[kFirst ? 1 : kPartItems];
  uint32_t id[kFirst ? kPartItems : 1];
  // a tile's items: the next tile's are in flight while this tile's go out
  auto load = [&](int64_t base) {
#pragma unroll
    for (int j = 0; j < kPartItems; ++j) {
      const int64_t i = base + w0 + 32 * j + lane;
      if constexpr (kFirst) id[j] = i < end ? static_cast<uint32_t>(__ldcs(ids + i)) : 0u;
      else v[j] = i < end ? __ldcs(in + i) : 0ull;
    }
  };
  load(begin);
  for (int64_t base = begin; base < end; base += kPartTile) {
    const int n = static_cast<int>(end - base < kPartTile ? end - base : kPartTile);
    for (int i = 8 * static_cast<int>(lane); i < n_digits; i += 256)
      *reinterpret_cast<uint4*>(&sm.wc[warp][i]) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    // the items' ranks within the warp and digit, in order
    uint32_t at[kPartItems];
#pragma unroll
    for (int j = 0; j < kPartItems; ++j) {
      const bool in_tile = w0 + 32 * j + static_cast<int>(lane) < n;
      uint32_t d = kPartNone;
      if (in_tile) {
        if constexpr (kFirst) d = id[j] >> lo_bits;
        else d = static_cast<uint32_t>(v[j] >> (kPartTrialBits + kPartKBits));
      }
      // Each lane puts its number in the digit's word and reads it back: the lanes whose number stands
      // there are alone with their digit or the one that the others see.  Few of 32 items share a digit,
      // so the shared ones are taken a digit at a time (with a warp match on every step instead, a
      // partition of 400M items took 5.2 ms against 3.6 ms, half its cycles in the unit that matches).
      uint32_t have = in_tile ? (sm.wc[warp][d] & kPartCntMask) : 0u;
      __syncwarp();
      if (in_tile) sm.wc[warp][d] = static_cast<uint16_t>((have + 1u) | (lane << kPartCntBits));
      __syncwarp();
      const uint32_t seen = in_tile ? (sm.wc[warp][d] >> kPartCntBits) : lane;
      uint32_t shared = __ballot_sync(0xffffffffu, seen != lane);
      uint32_t before = 0u;
      while (shared) {
        const uint32_t ds = __shfl_sync(0xffffffffu, d, __ffs(shared) - 1);
        const uint32_t peers = __ballot_sync(0xffffffffu, d == ds);
        if (d == ds) {
          before = __popc(peers & lt);
          if (before == 0u) sm.wc[warp][d] = static_cast<uint16_t>(have + __popc(peers));
        }
        shared &= ~peers;
      }
      __syncwarp();
      at[j] = (d << 16) | (have + before);
    }
    __syncthreads();
    // a thread's digits: counts over the warps to first places, over the digits too
    // (two digits a word: a tile's counts fit 16 bits)
    {
      constexpr int kW = kPartDigits / kPartThreads / 2;  // words a thread
      const uint32_t d0 = 2u * kW * tid;
      const bool mine = static_cast<int>(d0) < n_digits;
      uint32_t t[kW];
#pragma unroll
      for (int q = 0; q < kW; ++q) t[q] = 0u;
      if (mine) {
#pragma unroll
        for (int w = 0; w < kPartWarps; ++w) {
          uint32_t* p = reinterpret_cast<uint32_t*>(&sm.wc[w][d0]);
#pragma unroll
          for (int q = 0; q < kW; ++q) {
            const uint32_t c = p[q];
            p[q] = t[q];
            t[q] += c & (kPartCntMask | (kPartCntMask << 16));
          }
        }
      }
      uint32_t total = 0u;
#pragma unroll
      for (int q = 0; q < kW; ++q) total += (t[q] & 0xFFFFu) + (t[q] >> 16);
      uint32_t incl = total;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, s);
        if (lane >= static_cast<uint32_t>(s)) incl += o;
      }
      if (lane == 31u) sm.wsum[warp] = incl;
      __syncthreads();
      uint32_t first = incl - total;
      for (uint32_t w = 0; w < warp; ++w) first += sm.wsum[w];
      if (mine) {
        uint32_t add[kW];
#pragma unroll
        for (int q = 0; q < kW; ++q) {
          const uint32_t c0 = t[q] & 0xFFFFu, c1 = t[q] >> 16, d = d0 + 2u * q;
          const uint32_t r0 = sm.run[d], r1 = sm.run[d + 1];
          sm.gb[d] = r0 - first;
          sm.gb[d + 1] = r1 - (first + c0);
          sm.run[d] = r0 + c0;
          sm.run[d + 1] = r1 + c1;
          add[q] = first | ((first + c0) << 16);
          first += c0 + c1;
        }
#pragma unroll
        for (int w = 0; w < kPartWarps; ++w) {
          uint32_t* p = reinterpret_cast<uint32_t*>(&sm.wc[w][d0]);
#pragma unroll
          for (int q = 0; q < kW; ++q) p[q] += add[q];
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPartItems; ++j) {
      const uint32_t d = at[j] >> 16;
      if (d != kPartNone) at[j] += sm.wc[warp][d];  // below 2^16: the place in the tile
    }
    __syncthreads();  // dig shares wc's memory
    if constexpr (kFirst) {
      if (w0 < n) {
        tw = warp_trial_of(off, n_trials, tw, base + w0, lane);
        int64_t t = tw, cur = __ldg(off + t), next = __ldg(off + t + 1);
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) {
          const uint32_t d = at[j] >> 16;
          if (d == kPartNone) continue;
          const int64_t pos = base + w0 + 32 * j + lane;
          if (pos >= next) {
            for (int c = 0; pos >= next && c < 16; ++c) next = __ldg(off + (++t) + 1);
            if (pos >= next) {  // many short trials: the first b with off[b + 1] > pos
              int64_t a = t + 1, b = n_trials - 1;
              while (a < b) {
                const int64_t m = a + (b - a) / 2;
                if (__ldg(off + m + 1) > pos) b = m;
                else a = m + 1;
              }
              t = a;
              next = __ldg(off + t + 1);
            }
            cur = __ldg(off + t);
          }
          const uint32_t place = at[j] & 0xFFFFu;
          sm.stage[place] =
              (static_cast<unsigned long long>(id[j] & ((1u << lo_bits) - 1u)) << (kPartTrialBits + kPartKBits)) |
              (static_cast<unsigned long long>(t) << kPartKBits) | static_cast<unsigned long long>(pos - cur);
          sm.dig[place] = static_cast<uint16_t>(d);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < kPartItems; ++j) {
        const uint32_t d = at[j] >> 16;
        if (d == kPartNone) continue;
        const uint32_t place = at[j] & 0xFFFFu;
        sm.stage[place] = (((v[j] >> kPartKBits) & ((1ull << kPartTrialBits) - 1ull)) << 32) |
                          (v[j] & ((1ull << kPartKBits) - 1ull));
        sm.dig[place] = static_cast<uint16_t>(d);
      }
    }
    load(base + kPartTile);
    __syncthreads();
#pragma unroll 8
    for (int i = static_cast<int>(tid); i < n; i += kPartThreads)
      out[sm.gb[sm.dig[i]] + static_cast<uint32_t>(i)] = sm.stage[i];
    __syncthreads();
  }
}

// segment s of n_seg: YET positions [s E / n_seg, (s + 1) E / n_seg)
__device__ __forceinline__ int64_t part_bound(int64_t n_events, int n_seg, int64_t s) {
  return n_events / n_seg * s + n_events % n_seg * s / n_seg;
}

// cnt[d * n_seg + s]: the segment's events of each high digit (a CTA per segment)
__global__ void __launch_bounds__(1024) k_part_count(const int32_t* __restrict__ ids, int64_t n_events, int n_seg,
                                                     int lo_bits, int n_digits, uint32_t* cnt) {
  __shared__ uint32_t h[kPartDigits];
  for (int d = threadIdx.x; d < n_digits; d += blockDim.x) h[d] = 0u;
  __syncthreads();
  const int64_t end = part_bound(n_events, n_seg, blockIdx.x + 1);
  constexpr int kU = 8;  // loads in flight
  for (int64_t i = part_bound(n_events, n_seg, blockIdx.x) + threadIdx.x; i < end; i += kU * 1024) {
    int32_t e[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) e[u] = i + u * 1024 < end ? __ldcs(ids + i + u * 1024) : -1;
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (e[u] >= 0) atomicAdd(&h[e[u] >> lo_bits], 1u);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < n_digits; d += blockDim.x) cnt[static_cast<int64_t>(d) * n_seg + blockIdx.x] = h[d];
}

// The occurrences of the largest high digit's bucket (one block)
__global__ void __launch_bounds__(1024) k_part_largest(const uint32_t* __restrict__ start, int n_seg, int n_digits,
                                                       uint32_t* out) {
  __shared__ uint32_t most;
  if (threadIdx.x == 0) most = 0u;
  __syncthreads();
  for (int d = threadIdx.x; d < n_digits; d += blockDim.x)
    atomicMax(&most, start[static_cast<int64_t>(d + 1) * n_seg] - start[static_cast<int64_t>(d) * n_seg]);
  __syncthreads();
  if (threadIdx.x == 0) *out = most;
}

__global__ void __launch_bounds__(kPartThreads, 1)
    k_part_first(const int64_t* __restrict__ off, const int32_t* __restrict__ ids, int64_t n_trials, int64_t n_events,
                 int n_seg, int lo_bits, int n_digits, const uint32_t* __restrict__ start,
                 unsigned long long* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char part_smem[];
  PartShared& sm = *reinterpret_cast<PartShared*>(part_smem);
  for (int d = threadIdx.x; d < n_digits; d += kPartThreads)
    sm.run[d] = start[static_cast<int64_t>(d) * n_seg + blockIdx.x];
  __syncthreads();
  partition_items<true>(sm, off, ids, n_trials, lo_bits, nullptr, part_bound(n_events, n_seg, blockIdx.x),
                        part_bound(n_events, n_seg, blockIdx.x + 1), n_digits, out);
}

// A bucket's occurrences counted per (event, grid cell) into cnt (with the
// zero of each event's end column)
__global__ void __launch_bounds__(1024) k_part_cells(const unsigned long long* __restrict__ in, int n_seg, int lo_bits,
                                                     const uint32_t* __restrict__ start, int32_t catalogue,
                                                     int64_t cells, int grid_shift, uint32_t* __restrict__ cnt) {
  extern __shared__ __align__(16) uint32_t cell_cnt[];
  const int nc = static_cast<int>(cells);
  const int64_t e0 = static_cast<int64_t>(blockIdx.x) << lo_bits;
  const int n_ev = static_cast<int>(min(static_cast<int64_t>(catalogue) - e0, int64_t{1} << lo_bits));
  for (int i = threadIdx.x; i < n_ev * nc; i += blockDim.x) cell_cnt[i] = 0u;
  __syncthreads();
  const uint32_t a = start[static_cast<int64_t>(blockIdx.x) * n_seg];
  const uint32_t b = start[static_cast<int64_t>(blockIdx.x + 1) * n_seg];
  constexpr int kU = 4;
  // (64-bit positions: a may lie within a block of 2^32)
  for (uint64_t i = static_cast<uint64_t>(a) + threadIdx.x; i < b; i += kU * 1024) {
    unsigned long long v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = i + u * 1024 < b ? __ldcs(in + i + u * 1024) : ~0ull;
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (i + u * 1024 < b) {
        const uint32_t el = static_cast<uint32_t>(v[u] >> (kPartTrialBits + kPartKBits));
        const uint32_t t = static_cast<uint32_t>(v[u] >> kPartKBits) & ((1u << kPartTrialBits) - 1u);
        atomicAdd(&cell_cnt[el * nc + (t >> grid_shift)], 1u);
      }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n_ev * (nc + 1); i += blockDim.x) {
    const int el = i / (nc + 1), c = i - el * (nc + 1);
    cnt[e0 * (nc + 1) + i] = c < nc ? cell_cnt[el * nc + c] : 0u;
  }
}

__global__ void __launch_bounds__(kPartThreads, 1)
    k_part_second(const unsigned long long* __restrict__ in, int n_seg, int lo_bits, const uint32_t* __restrict__ start,
                  int32_t catalogue, int64_t cells1, const uint32_t* __restrict__ ev_grid,
                  unsigned long long* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char part_smem[];
  PartShared& sm = *reinterpret_cast<PartShared*>(part_smem);
  const int64_t e0 = static_cast<int64_t>(blockIdx.x) << lo_bits;
  const int n_ev = static_cast<int>(min(static_cast<int64_t>(catalogue) - e0, int64_t{1} << lo_bits));
  const int64_t begin = start[static_cast<int64_t>(blockIdx.x) * n_seg];
  const int64_t end = start[static_cast<int64_t>(blockIdx.x + 1) * n_seg];
  if (begin >= end) return;
  for (int d = threadIdx.x; d < n_ev; d += kPartThreads) sm.run[d] = ev_grid[(e0 + d) * cells1];
  __syncthreads();
  partition_items<false>(sm, nullptr, nullptr, 0, lo_bits, in, begin, end, n_ev, out);
}

constexpr int64_t kScatterEvents = int64_t{1} << 18;  // events a scatter pass places

int grid_of(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return static_cast<int>(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

}  // namespace

int64_t yet_grid_cells(int64_t n_trials, int grid_shift) {
  return n_trials > 0 ? ((n_trials - 1) >> grid_shift) + 1 : 0;
}

size_t yet_bucket_scratch_bytes(int32_t catalogue, int64_t cells) {
  const int64_t n = static_cast<int64_t>(catalogue) * (cells + 1);
  return sizeof(uint32_t) * (static_cast<size_t>(n) + scan_tmp_words(n) + 64);
}

cudaError_t yet_index_count(const int64_t* off, const int32_t* ids, int64_t n_trials, int32_t catalogue, int grid_shift,
                            uint32_t* ev_grid, void* scratch, cudaStream_t s, int* n_launch) {
  const int64_t cells1 = yet_grid_cells(n_trials, grid_shift) + 1;
  const int64_t n = static_cast<int64_t>(catalogue) * cells1;
  uint32_t* cnt = static_cast<uint32_t*>(scratch);
  uint32_t* d_max = cnt + n;
  uint32_t* tmp = d_max + 32;
  cudaError_t err = cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * (static_cast<size_t>(n) + 32), s);
  if (err != cudaSuccess) return err;
  if (n_trials > 0) {
    k_count_cells<<<grid_of(n_trials * 32, 256), 256, 0, s>>>(off, ids, n_trials, cells1, grid_shift, cnt);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    if (n_launch) ++*n_launch;
  }
  k_max_u32<<<grid_of(n, 256), 256, 0, s>>>(cnt, n, d_max);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if (n_launch) ++*n_launch;
  return scan_exclusive_u32(cnt, ev_grid, n, tmp, s, n_launch);
}

const uint32_t* yet_index_max_bucket(const void* scratch, int32_t catalogue, int64_t cells) {
  return static_cast<const uint32_t*>(scratch) + static_cast<int64_t>(catalogue) * (cells + 1);
}

cudaError_t yet_index_fill(const int64_t* off, const int32_t* ids, int64_t n_trials, int32_t catalogue, int grid_shift,
                           const uint32_t* ev_grid, unsigned long long* occ, void* scratch, cudaStream_t s,
                           int* n_launch) {
  const int64_t cells1 = yet_grid_cells(n_trials, grid_shift) + 1;
  const int64_t n = static_cast<int64_t>(catalogue) * cells1;
  uint32_t* cur = static_cast<uint32_t*>(scratch);
  cudaError_t err = cudaMemsetAsync(cur, 0, sizeof(uint32_t) * static_cast<size_t>(n), s);
  if (err != cudaSuccess || n_trials <= 0) return err;
  int launched = 1;
  for (int64_t e_lo = 0; e_lo < catalogue; e_lo += kScatterEvents, ++launched) {
    const int32_t e_hi = static_cast<int32_t>(e_lo + kScatterEvents < catalogue ? e_lo + kScatterEvents : catalogue);
    k_scatter_cells<<<grid_of(n_trials * 32, 256), 256, 0, s>>>(off, ids, n_trials, cells1, grid_shift,
                                                               static_cast<int32_t>(e_lo), e_hi, ev_grid, cur, occ);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  k_sort_cells<<<grid_of(n, 256), 256, 0, s>>>(ev_grid, n, occ);
  if (n_launch) *n_launch += launched;
  return cudaGetLastError();
}

namespace {

// The partition build's shape.  The high digit takes the bits that leave
// buckets of about one tile or more (at least 256 of them, so that every SM
// has some), the low digit the rest; each at most 11 bits.
struct PartShape {
  int lo_bits, n_digits, n_seg;
};

PartShape part_shape(int64_t n_events, int32_t catalogue, int num_sms) {
  int bits = 1;
  while (bits < 31 && (int64_t{1} << bits) < static_cast<int64_t>(catalogue)) ++bits;
  int hi = 8;
  while (hi < 11 && (n_events >> hi) > kPartTile) ++hi;
  PartShape sh;
  sh.lo_bits = bits - hi < 1 ? 1 : bits - hi > 11 ? 11 : bits - hi;
  sh.n_digits = static_cast<int>(((catalogue - 1) >> sh.lo_bits) + 1);
  const int64_t tiles = (n_events + kPartTile - 1) / kPartTile;
  const int64_t most = int64_t{4} * num_sms;  // four segments an SM even out the last ones
  sh.n_seg = static_cast<int>(tiles < 1 ? 1 : tiles < most ? tiles : most);
  return sh;
}

constexpr size_t kPartCellBytes = 200 * 1024;  // shared memory of k_part_cells, at most

// A bucket of the first partition goes to one CTA, so the build waits for the largest.  The partitions are
// taken while that has at most a 32nd of the events (five times an SM's share), or no more than the bucket
// build would sort with a thread.  100M events over 10,000 ids, one of them with 2% and 3% of all: 2.9 and 3.8
// ms, by the radix sort 9.6 and 9.6; they meet near 20% (18.9 and 19.9 ms).
constexpr int64_t kPartUneven = 32;
constexpr uint32_t kPartSmall = 2048;

}  // namespace

// Whether the bucket build is the faster one: its launches are cheaper, while few occurrences of an event share
// a bucket and the events are too few to fill the SMs, or the catalogue's counts are small.  us by buckets and
// by partitions: 100,000 events over 20,000 ids 64 and 108, 1M over 200,000 95 and 123, 3M over 200,000 142 and
// 157, 20,000 over 2,000,000 148 and 159; but 1M over 20,000 187 and 147, 10M over 200,000 363 and 337, 100,000
// over 2,000,000 182 and 172.
static bool few_events(int64_t n_events, int32_t catalogue) {
  return n_events <= (int64_t{3} << 20) && n_events <= 16 * static_cast<int64_t>(catalogue) &&
         (catalogue <= (1 << 19) || n_events < (1 << 15));
}

bool yet_parts_fit(int64_t n_trials, int64_t n_events, int32_t catalogue, int64_t cells, int num_sms) {
  const PartShape sh = part_shape(n_events, catalogue, num_sms);
  return n_events > 0 && !few_events(n_events, catalogue) && n_events < (int64_t{1} << 32) - 1 && n_trials <= (int64_t{1} << kPartTrialBits) &&
         sh.n_digits <= kPartDigits && sizeof(uint32_t) * (static_cast<size_t>(cells) << sh.lo_bits) <= kPartCellBytes;
}

size_t yet_parts_scratch_bytes(int64_t n_events, int32_t catalogue, int64_t cells, int num_sms) {
  const PartShape sh = part_shape(n_events, catalogue, num_sms);
  const int64_t np = static_cast<int64_t>(sh.n_digits) * sh.n_seg, n = static_cast<int64_t>(catalogue) * (cells + 1);
  return sizeof(uint32_t) * (64 + 2 * static_cast<size_t>(np) + 1 + static_cast<size_t>(n) +
                             (scan_tmp_words(np) > scan_tmp_words(n) ? scan_tmp_words(np) : scan_tmp_words(n)));
}

namespace {

// scratch: the largest bucket's count (in 32 words), the segments' digit
// counts, their scan, the (event, cell) counts, the scans' scratch
struct PartScratch {
  uint32_t *largest, *seg_cnt, *start, *cnt, *tmp;
};

PartScratch part_scratch(void* scratch, const PartShape& sh, int32_t catalogue, int64_t cells) {
  const int64_t np = static_cast<int64_t>(sh.n_digits) * sh.n_seg;
  PartScratch p;
  p.largest = static_cast<uint32_t*>(scratch);
  p.seg_cnt = p.largest + 32;
  p.start = p.seg_cnt + np;
  p.cnt = p.start + np + 1;
  p.tmp = p.cnt + static_cast<int64_t>(catalogue) * (cells + 1);
  return p;
}

}  // namespace

cudaError_t yet_parts_count(const int32_t* ids, int64_t n_events, int32_t catalogue, int64_t cells, int num_sms,
                            void* scratch, cudaStream_t s, int* n_launch) {
  const PartShape sh = part_shape(n_events, catalogue, num_sms);
  const PartScratch p = part_scratch(scratch, sh, catalogue, cells);
  k_part_count<<<sh.n_seg, 1024, 0, s>>>(ids, n_events, sh.n_seg, sh.lo_bits, sh.n_digits, p.seg_cnt);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if ((err = scan_exclusive_u32(p.seg_cnt, p.start, static_cast<int64_t>(sh.n_digits) * sh.n_seg, p.tmp, s,
                                n_launch)) != cudaSuccess)
    return err;
  k_part_largest<<<1, 1024, 0, s>>>(p.start, sh.n_seg, sh.n_digits, p.largest);
  if (n_launch) *n_launch += 2;
  return cudaGetLastError();
}

int64_t yet_parts_bucket_ids(int64_t n_events, int32_t catalogue, int num_sms) {
  return int64_t{1} << part_shape(n_events, catalogue, num_sms).lo_bits;
}

bool yet_parts_even(uint32_t largest, int64_t n_events) {
  return largest <= kPartSmall || static_cast<int64_t>(largest) * kPartUneven <= n_events;
}

cudaError_t yet_parts_first(const int64_t* off, const int32_t* ids, int64_t n_trials, int64_t n_events,
                            int32_t catalogue, int grid_shift, int num_sms, unsigned long long* parts,
                            uint32_t* ev_grid, void* scratch, cudaStream_t s, int* n_launch) {
  const int64_t cells = yet_grid_cells(n_trials, grid_shift);
  const PartShape sh = part_shape(n_events, catalogue, num_sms);
  const PartScratch p = part_scratch(scratch, sh, catalogue, cells);
  const int smem = static_cast<int>(sizeof(PartShared));
  const int cell_smem = static_cast<int>(sizeof(uint32_t) * (static_cast<size_t>(cells) << sh.lo_bits));
  cudaError_t err;
  if ((err = cudaFuncSetAttribute(k_part_first, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess ||
      // (the limit belongs to the function: the most that any build asks for, as contexts on other threads
      // launch it too)
      (err = cudaFuncSetAttribute(k_part_cells, cudaFuncAttributeMaxDynamicSharedMemorySize, kPartCellBytes)) !=
          cudaSuccess)
    return err;
  k_part_first<<<sh.n_seg, kPartThreads, smem, s>>>(off, ids, n_trials, n_events, sh.n_seg, sh.lo_bits, sh.n_digits,
                                                   p.start, parts);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  k_part_cells<<<sh.n_digits, 1024, cell_smem, s>>>(parts, sh.n_seg, sh.lo_bits, p.start, catalogue, cells, grid_shift,
                                                   p.cnt);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if (n_launch) *n_launch += 2;
  return scan_exclusive_u32(p.cnt, ev_grid, static_cast<int64_t>(catalogue) * (cells + 1), p.tmp, s, n_launch);
}

cudaError_t yet_parts_fill(int64_t n_trials, int64_t n_events, int32_t catalogue, int grid_shift, int num_sms,
                           const unsigned long long* parts, const uint32_t* ev_grid, unsigned long long* occ,
                           void* scratch, cudaStream_t s, int* n_launch) {
  const int64_t cells = yet_grid_cells(n_trials, grid_shift);
  const PartShape sh = part_shape(n_events, catalogue, num_sms);
  const PartScratch p = part_scratch(scratch, sh, catalogue, cells);
  const int smem = static_cast<int>(sizeof(PartShared));
  const cudaError_t err = cudaFuncSetAttribute(k_part_second, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (err != cudaSuccess) return err;
  k_part_second<<<sh.n_digits, kPartThreads, smem, s>>>(parts, sh.n_seg, sh.lo_bits, p.start, catalogue, cells + 1,
                                                       ev_grid, occ);
  if (n_launch) *n_launch += 1;
  return cudaGetLastError();
}

size_t yet_index_scratch_bytes(int64_t n_events, int32_t catalogue) {
  return sizeof(unsigned long long) * static_cast<size_t>(n_events) + sort_pairs_scratch_bytes(n_events) +
         sizeof(uint32_t) * (static_cast<size_t>(catalogue) + 2) + 512;
}

cudaError_t build_yet_index(const int64_t* off, const int32_t* ids, int64_t n_trials, int64_t n_events,
                            int32_t catalogue, int grid_shift, unsigned long long* occ, uint32_t* ev_grid,
                            void* scratch, cudaStream_t s, int* n_launch) {
  unsigned long long* keys = static_cast<unsigned long long*>(scratch);
  uint32_t* ev_off = reinterpret_cast<uint32_t*>(keys + n_events);  // [catalogue + 1]
  void* sort_scratch = reinterpret_cast<char*>(scratch) + sizeof(unsigned long long) * static_cast<size_t>(n_events) +
                       ((sizeof(uint32_t) * (static_cast<size_t>(catalogue) + 2) + 255) & ~size_t{255});
  const int64_t cells = yet_grid_cells(n_trials, grid_shift);
  const int64_t n_entries = static_cast<int64_t>(catalogue) * (cells + 1);
  k_fill_u32<<<grid_of(static_cast<int64_t>(catalogue) + 1, 256), 256, 0, s>>>(ev_off, static_cast<int64_t>(catalogue) + 1,
                                                                              static_cast<uint32_t>(n_events));
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  int launched = 1;
  if (n_events > 0) {
    k_yet_pairs<<<grid_of(n_trials * 32, 256), 256, 0, s>>>(off, ids, n_trials, keys, reinterpret_cast<int64_t*>(occ));
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    int key_bits = 1;
    while (key_bits < 31 && (1ll << key_bits) < static_cast<int64_t>(catalogue)) ++key_bits;
    if ((err = sort_pairs_ascending(keys, reinterpret_cast<int64_t*>(occ), n_events, key_bits, sort_scratch, s,
                                    n_launch)) != cudaSuccess)
      return err;
    k_event_starts<<<grid_of(n_events, 256), 256, 0, s>>>(keys, n_events, ev_off);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    launched += 2;
  }
  if (n_entries > 0) {
    k_event_grid<<<grid_of(n_entries, 256), 256, 0, s>>>(occ, ev_off, n_entries, cells, grid_shift, ev_grid);
    ++launched;
  }
  if (n_launch) *n_launch += launched;
  return cudaGetLastError();
}

}  // namespace ara
