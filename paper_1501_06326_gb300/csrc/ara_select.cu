// PML / TVaR (Section 2.3) and the YLT trial order on the device.
//
// Year losses are mapped to order-preserving 64-bit keys (sign-flipped IEEE
// bits).  PML(RP) is the m-th largest year loss, m = ceil(n / RP): an MSB-first
// radix select narrows the key's bits, 11 at a time.  TVaR(RP) is the mean of
// the m largest: the sum of the values whose key exceeds the m-th key plus the
// tied remainder times the m-th value, in FP64 with a fixed assignment of
// values to threads and a fixed reduction order (deterministic).  The full
// trial order (largest first, ties by index) is a stable LSD radix sort of the
// complemented keys.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdint>
#include <utility>

#include "../../include/ara.h"
#include "ara_batch.h"

namespace ara {

namespace {

namespace cg = cooperative_groups;

__device__ __forceinline__ unsigned long long key_of(double v) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double value_of(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
  return __longlong_as_double(static_cast<long long>(b));
}

// k_select: one thread-block cluster per job (a YLT and up to four return
// periods), in one launch and without scratch in device memory.  Value i of
// the YLT belongs to thread i mod (CTAs x 1,024) of the cluster.  Two passes
// count a digit of 11 bits (sign, exponent, 11 bits of the significand: the
// key's upper half) among the keys that match a period's prefix, in shared
// memory; the CTAs' counts are added through distributed shared memory, and
// every CTA picks each period's next digit.  The keys that then match a prefix
// are collected.  When the cluster has at most kSelFew of them, each CTA ranks
// them all against one another; when values are tied there are more, and four
// digits follow over the collected keys (or the YLT, where a CTA's own do not
// fit).  A last pass sums the values above each m-th key.
// A short YLT is bound by the chain of passes and its barriers, and by the
// instruction cache, as the code runs once (hence the loops that are not
// unrolled and sel_pick not inlined: 41 us inlined, 1,000 trials); a long one by
// one GPC's 16 SMs passing over it four times.  Device time at 1,000 / 20,000 /
// 1,000,000 trials and two periods: 21 / 29 / 63 us; five launches with
// histograms in device memory took 60 / 66 / 95 us, and an occurrence YLT with
// 100,000 tied values 167 us against 65.
constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelUnroll = 8;     // loads in flight per thread
constexpr int kSelGroup = 4;      // return periods selected together
constexpr int kSelBatchMax = 32;  // jobs of one launch
constexpr int kSelBins = 2048;
constexpr int kSelList = 8192;    // keys a CTA collects
constexpr int kSelFew = 256;      // keys of a cluster that are ranked directly, at most

struct SelJob {
  const double* ylt;
  int64_t n;
  double* pml;
  double* tvar;               // or NULL: no sums
  unsigned long long* ties;   // or NULL: of the m-th value's ties, how many are among the m largest
  unsigned long long m[kSelGroup];
  int g;
};
struct SelBatch {
  SelJob job[kSelBatchMax];
};

struct SelShared {
  union {
    unsigned int hist[kSelGroup][kSelBins];   // this CTA's counts
    unsigned long long ring[kSelWarps][64];   // the last pass: keys to be summed, per warp
    unsigned long long few[kSelFew];          // the cluster's collected keys, when they are few
  };
  unsigned int total[kSelGroup][kSelBins];    // the cluster's counts
  unsigned long long list[kSelList];          // collected keys
  unsigned int n_list;
  unsigned int warp_sum[kSelWarps];
  // per period: the key's bits fixed so far, the rank wanted among the keys with them (1 = largest)
  unsigned long long prefix[kSelGroup], want[kSelGroup];
  double part[kSelWarps][kSelGroup];
  double cta_sum[kSelGroup];
};

// The values of the YLT that belong to this thread (kStride apart): f(value,
// valid) is called by whole warps.
template <int kStride, class F>
__device__ __forceinline__ void sel_values(const SelJob& j, int first, F f) {
  const double* p = j.ylt + first;
  const int64_t left = j.n - first;
  const int64_t cnt = left > 0 ? (left + kStride - 1) / kStride : 0;
  const int64_t most = __shfl_sync(0xffffffffu, cnt, 0);  // the warp's first lane has the most
#pragma unroll 1
  for (int64_t u0 = 0; u0 < most; u0 += kSelUnroll, p += static_cast<int64_t>(kSelUnroll) * kStride) {
    const int here = static_cast<int>(cnt - u0 < kSelUnroll ? cnt - u0 : kSelUnroll);
    double v[kSelUnroll];
#pragma unroll
    for (int u = 0; u < kSelUnroll; ++u) v[u] = u < here ? p[static_cast<int64_t>(u) * kStride] : 0.0;
#pragma unroll
    for (int u = 0; u < kSelUnroll; ++u) f(v[u], u < here);
  }
}

// The upper half of a value's key.
__device__ __forceinline__ unsigned int key_hi(double v) {
  const int h = __double2hiint(v);
  return static_cast<unsigned int>(h) ^ (static_cast<unsigned int>(h >> 31) | 0x80000000u);
}

// Whether period r is the first with its prefix (the others share its counts).
__device__ __forceinline__ bool sel_owns(const SelShared& sm, int g, int r) {
  bool own = r < g;
#pragma unroll
  for (int q = 0; q < kSelGroup; ++q) own = own && !(q < r && sm.prefix[q] == sm.prefix[r]);
  return own;
}

// Clears the counts (by all threads; ends with a barrier).
__device__ __noinline__ void sel_clear(SelShared& sm) {
  uint4* h = reinterpret_cast<uint4*>(&sm.hist[0][0]);
#pragma unroll
  for (int i = 0; i < kSelGroup * kSelBins / 4 / kSelThreads; ++i)
    h[i * kSelThreads + threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
}

// One digit of `bits` bits from its counts in sm.hist: their sums over the
// cluster, and each period's choice.  Not inlined: the kernel runs its code
// once, so the instruction cache's misses count.
template <int kCtas>
__device__ __noinline__ void sel_pick(SelShared& sm, int g, int bits) {
  const unsigned int t = threadIdx.x, lane = t & 31u, r = t >> 8, u = t & 255u;
  unsigned int* total = &sm.total[0][0];
  if constexpr (kCtas > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned int rank = cluster.block_rank();
    unsigned int* hist = &sm.hist[0][0];
    cluster.sync();
    // this CTA's share of the bins, summed over the cluster; then everyone's shares.  The r-th quarter of
    // the threads takes period r
    constexpr unsigned int kShare = kSelBins / kCtas;
    const bool own = sel_owns(sm, g, static_cast<int>(r));
    if (own)
#pragma unroll 1
      for (unsigned int i = rank * kShare + u; i < (rank + 1) * kShare; i += 256) {
        unsigned int s[kCtas], all = 0u;
#pragma unroll
        for (int c = 0; c < kCtas; ++c) s[c] = cluster.map_shared_rank(hist, c)[r * kSelBins + i];
#pragma unroll
        for (int c = 0; c < kCtas; ++c) all += s[c];
        total[r * kSelBins + i] = all;
      }
    cluster.sync();
    if (own)
#pragma unroll
      for (unsigned int i = u; i < kSelBins; i += 256) {
        const unsigned int c = i / kShare;
        if (c != rank) total[r * kSelBins + i] = cluster.map_shared_rank(total, c)[r * kSelBins + i];
      }
  } else {
    total = &sm.hist[0][0];
  }
  __syncthreads();
  // period r's digit, 8 bins a thread from the top: the first whose running count reaches the wanted rank
  const bool live = static_cast<int>(r) < g;
  unsigned int c[8], sum = 0u;
  if (live) {
    int slot = static_cast<int>(r);
#pragma unroll
    for (int q = kSelGroup - 1; q >= 0; --q)
      if (q < static_cast<int>(r) && sm.prefix[q] == sm.prefix[r]) slot = q;
    const uint4* tk = reinterpret_cast<const uint4*>(total + slot * kSelBins + (kSelBins - 8 - 8 * u));
    const uint4 lo = tk[0], hi = tk[1];  // a digit of fewer bits leaves its upper bins empty
    c[0] = hi.w; c[1] = hi.z; c[2] = hi.y; c[3] = hi.x;
    c[4] = lo.w; c[5] = lo.z; c[6] = lo.y; c[7] = lo.x;
#pragma unroll
    for (int q = 0; q < 8; ++q) sum += c[q];
  }
  unsigned int incl = sum;
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, incl, dd);
    if (lane >= static_cast<unsigned int>(dd)) incl += o;
  }
  if (lane == 31u) sm.warp_sum[t >> 5] = incl;
  const unsigned long long want = live ? sm.want[r] : 0ull;
  __syncthreads();
  unsigned long long before = incl - sum;
#pragma unroll
  for (unsigned int w = 0; w < 7; ++w)
    if (w < ((t >> 5) & 7u)) before += sm.warp_sum[r * 8 + w];
  if (live && before < want && want <= before + sum) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (before < want && want <= before + c[q]) {
        sm.want[r] = want - before;
        sm.prefix[r] = (sm.prefix[r] << bits) | (kSelBins - 1 - (8 * u + q));
      }
      before += c[q];
    }
  }
  __syncthreads();
}

// Per period the sum of this thread's values above its key kth.  A warp
// collects the values above the lowest of the keys in its ring of 64 and adds 32
// at a time, as an FP64 add costs a whole warp's time however few lanes need it.
template <int kStride>
__device__ __forceinline__ void sel_sums(const SelJob& j, int first, const unsigned long long (&kth)[kSelGroup],
                                         unsigned long long* ring, double (&sum)[kSelGroup]) {
  const unsigned int lane = threadIdx.x & 31u;
  unsigned long long lowest = ~0ull;
#pragma unroll
  for (int r = 0; r < kSelGroup; ++r) {
    sum[r] = 0.0;
    lowest = kth[r] < lowest ? kth[r] : lowest;
  }
  const unsigned int lowest_hi = static_cast<unsigned int>(lowest >> 32);
  unsigned int held = 0u;
  auto add = [&](unsigned long long key, bool valid) {
    const double v = value_of(key);
#pragma unroll
    for (int r = 0; r < kSelGroup; ++r)
      if (valid && key > kth[r]) sum[r] += v;
  };
  sel_values<kStride>(j, first, [&](double v, bool valid) {
    bool above = valid && key_hi(v) >= lowest_hi;
    if (__ballot_sync(0xffffffffu, above) == 0u) return;
    const unsigned long long key = key_of(v);
    above = above && key > lowest;
    const unsigned int mm = __ballot_sync(0xffffffffu, above);
    if (above) ring[held + __popc(mm & ((1u << lane) - 1u))] = key;
    held += __popc(mm);
    __syncwarp();
    if (held >= 32u) {
      add(ring[lane], true);
      held -= 32u;
      const unsigned long long rest = ring[32 + lane];
      __syncwarp();
      ring[lane] = rest;
      __syncwarp();
    }
  });
  add(lane < held ? ring[lane] : 0ull, lane < held);
}

template <int kCtas>
__global__ void __launch_bounds__(kSelThreads, 1) k_select(const __grid_constant__ SelBatch b) {
  extern __shared__ __align__(16) unsigned char sel_smem[];
  SelShared& sm = *reinterpret_cast<SelShared*>(sel_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const SelJob& j = b.job[blockIdx.y];
  constexpr int kStride = kCtas * kSelThreads;
  const unsigned int t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const unsigned int rank = kCtas > 1 ? cluster.block_rank() : 0u;
  const int first = static_cast<int>(rank * kSelThreads + t);
  if (t < static_cast<unsigned int>(kSelGroup)) {
    sm.prefix[t] = 0ull;
    sm.want[t] = j.m[t];
  }
  if (t == 0) sm.n_list = 0u;
  sel_clear(sm);
  // the first two digits are in the key's upper half; with nothing fixed there is one set of counts
  sel_values<kStride>(j, first, [&](double v, bool valid) {
    if (valid) atomicAdd(&sm.hist[0][key_hi(v) >> 21], 1u);
  });
  __syncthreads();
  sel_pick<kCtas>(sm, j.g, 11);
  unsigned int p32[kSelGroup];
#pragma unroll
  for (int k = 0; k < kSelGroup; ++k) p32[k] = sel_owns(sm, j.g, k) ? static_cast<unsigned int>(sm.prefix[k]) : ~0u;
  sel_clear(sm);
  sel_values<kStride>(j, first, [&](double v, bool valid) {
    const unsigned int h = key_hi(v), top = valid ? h >> 21 : ~0u - 1u;
#pragma unroll
    for (int k = 0; k < kSelGroup; ++k)
      if (top == p32[k]) atomicAdd(&sm.hist[k][(h >> 10) & 2047u], 1u);
  });
  __syncthreads();
  sel_pick<kCtas>(sm, j.g, 11);
  // the keys that still match, where this CTA has room for its own
#pragma unroll
  for (int k = 0; k < kSelGroup; ++k) p32[k] = k < j.g ? static_cast<unsigned int>(sm.prefix[k]) : ~0u;
  sel_values<kStride>(j, first, [&](double v, bool valid) {
    const unsigned int top = valid ? key_hi(v) >> 10 : ~0u - 1u;
    const bool match = top == p32[0] || top == p32[1] || top == p32[2] || top == p32[3];
    const unsigned int mm = __ballot_sync(0xffffffffu, match);
    if (mm == 0u) return;
    unsigned int at = 0u;
    if (lane == 0) at = atomicAdd(&sm.n_list, static_cast<unsigned int>(__popc(mm)));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(mm & ((1u << lane) - 1u));
    if (match && at < kSelList) sm.list[at] = key_of(v);
  });
  // few in the whole cluster: every CTA takes them all and ranks them
  unsigned int n_few = 0u;
  if constexpr (kCtas > 1) cluster.sync();
  else __syncthreads();
#pragma unroll
  for (int c = 0; c < kCtas; ++c) n_few += kCtas > 1 ? *cluster.map_shared_rank(&sm.n_list, c) : sm.n_list;
  if (n_few <= kSelFew) {
    if constexpr (kCtas > 1) {
      unsigned int at = 0u;
#pragma unroll 1
      for (int c = 0; c < kCtas; ++c) {
        const unsigned int n = *cluster.map_shared_rank(&sm.n_list, c);
        if (t < n) sm.few[at + t] = cluster.map_shared_rank(sm.list, c)[t];
        at += n;
      }
      __syncthreads();
    }
    const unsigned long long* few = kCtas > 1 ? sm.few : sm.list;
    unsigned long long want[kSelGroup];
#pragma unroll
    for (int r = 0; r < kSelGroup; ++r) want[r] = sm.want[r];
    if (kCtas > 1) cluster.sync();  // the lists are read
    else __syncthreads();
    if (t < n_few) {
      const unsigned long long mine = few[t], top = mine >> 42;
      unsigned int above = 0u, same = 0u;
#pragma unroll 4
      for (unsigned int i = 0; i < n_few; ++i) {
        const unsigned long long k = few[i];
        above += (k > mine && (k >> 42) == top) ? 1u : 0u;
        same += k == mine ? 1u : 0u;
      }
#pragma unroll
      for (int r = 0; r < kSelGroup; ++r)
        if (r < j.g && static_cast<unsigned int>(top) == p32[r] && above < want[r] && want[r] <= above + same) {
          sm.prefix[r] = mine;  // ties write the same
          sm.want[r] = want[r] - above;
        }
    }
    __syncthreads();
  } else {
    const bool from_list = sm.n_list <= kSelList;
#pragma unroll 1
    for (int shift = 31, bits = 11; shift >= 0; shift = shift == 31 ? 20 : shift - 10, bits = shift > 10 ? 11 : 10) {
      sel_clear(sm);
      unsigned long long own[kSelGroup];
#pragma unroll
      for (int k = 0; k < kSelGroup; ++k) own[k] = sel_owns(sm, j.g, k) ? sm.prefix[k] : ~0ull;
      auto count = [&](unsigned long long key, bool valid) {
        const unsigned int d = static_cast<unsigned int>(key >> shift) & ((1u << bits) - 1u);
        const unsigned long long top = valid ? key >> (shift + bits) : ~0ull - 1ull;
#pragma unroll
        for (int k = 0; k < kSelGroup; ++k)
          if (top == own[k]) atomicAdd(&sm.hist[k][d], 1u);
      };
      if (from_list) {
#pragma unroll 1
        for (unsigned int i = t; i < sm.n_list; i += kSelThreads) count(sm.list[i], true);
      } else {
        sel_values<kStride>(j, first, [&](double v, bool valid) { count(key_of(v), valid); });
      }
      __syncthreads();
      sel_pick<kCtas>(sm, j.g, bits);
    }
    if (kCtas > 1) cluster.sync();  // ring shares hist's memory, which the other CTAs have read by now
  }
  if (j.ties && rank == 0 && static_cast<int>(t) < j.g) j.ties[t] = sm.want[t];
  if (!j.tvar) {
    if (rank == 0 && static_cast<int>(t) < j.g) j.pml[t] = value_of(sm.prefix[t]);
    return;  // (no CTA reads another's shared memory any more)
  }
  // sums of the values above each period's key
  double sum[kSelGroup];
  unsigned long long kth[kSelGroup];
#pragma unroll
  for (int r = 0; r < kSelGroup; ++r) kth[r] = r < j.g ? sm.prefix[r] : ~0ull;
  __syncthreads();  // few shares ring's memory
  sel_sums<kStride>(j, first, kth, sm.ring[warp], sum);
#pragma unroll
  for (int r = 0; r < kSelGroup; ++r) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum[r] += __shfl_down_sync(0xffffffffu, sum[r], d);
    if (lane == 0) sm.part[warp][r] = sum[r];
  }
  __syncthreads();
  if (t < static_cast<unsigned int>(kSelGroup)) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) s += sm.part[w][t];
    sm.cta_sum[t] = s;
  }
  if (kCtas > 1) cluster.sync();
  else __syncthreads();
  if (rank == 0 && static_cast<int>(t) < j.g) {
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < kCtas; ++c) s += kCtas > 1 ? cluster.map_shared_rank(sm.cta_sum, c)[t] : sm.cta_sum[t];
    // want is now the m-th key's rank among its ties: the values above it number m - want
    const double v = value_of(sm.prefix[t]);
    j.pml[t] = v;
    j.tvar[t] = (s + static_cast<double>(sm.want[t]) * v) / static_cast<double>(j.m[t]);
  }
  if (kCtas > 1) cluster.sync();  // the CTAs' sums stay until they are read
}

// The wide select, for YLTs longer than kSelWide: all SMs pass over the YLT, in
// a launch for each digit and one for the sums.  A launch first picks the digit
// before it from its counts (every CTA the same), then counts its own in shared
// memory and adds the counts to the job's scratch.  Six digits of 11 bits (the
// last of 9); eight of 8 where the scratch must be small, with the same results.
// Up to about 1M values it is bound by the launches' latency (11 us each, 78 in
// all), a long YLT by reading it seven times (64M values, 512 MB: 5.2 TB/s).
constexpr int kWideCtas = 152;  // one an SM
constexpr int kWideBits = 11, kWideBitsSmall = 8;

template <int kBits>
struct WideScratch {
  static constexpr int kBins = 1 << kBits, kDigits = (64 + kBits - 1) / kBits;
  // counts of digit L in hist[of(L)]: the launch of digit L reads those of digit L - 1, adds its own and clears those
  // of digit L + 1; the last digit's are in hist[0], so that the sums' parts, [CTA][period], take the other two
  unsigned int hist[3][kSelGroup][kBins];
  __device__ static int of(int digit) { return (digit + 3 - (kDigits - 1) % 3) % 3; }
  __device__ double* parts() { return reinterpret_cast<double*>(&hist[1][0][0]); }
  unsigned long long prefix[2][kSelGroup], want[2][kSelGroup];  // after digit L: [L & 1]
  unsigned int done, pad;  // CTAs whose sums are there
  static_assert(2 * sizeof(unsigned int) * kSelGroup * kBins >= sizeof(double) * kWideCtas * kSelGroup, "parts fit");
};

struct WideBatch {
  SelJob job[kSelBatchMax];
  void* scratch;  // one a job
};

template <int kBits>
struct WideShared {
  unsigned int hist[kSelGroup][1 << kBits];
  unsigned int warp_sum[kSelWarps];
  unsigned long long prefix[kSelGroup], want[kSelGroup];
};

// Digit L is the key's bits [wide_shift(L), wide_shift(L) + its width).
template <int kBits>
__device__ __forceinline__ int wide_shift(int digit) {
  const int low = 64 - kBits * (digit + 1);
  return low > 0 ? low : 0;
}

// Picks each period's digit L from its counts (all threads, the r-th quarter period r; ends with a barrier).
template <int kBits>
__device__ __forceinline__ void wide_pick(const SelJob& j, WideScratch<kBits>& w, WideShared<kBits>& sm, int digit) {
  constexpr int kBins = 1 << kBits, kOwn = kBins / 256;  // bins of a thread
  const unsigned int t = threadIdx.x, lane = t & 31u, r = t >> 8, u = t & 255u;
  const bool live = static_cast<int>(r) < j.g;
  unsigned long long mine = 0ull, want = 0ull;
  unsigned int c[kOwn], sum = 0u;
  if (live) {
    unsigned int slot = r;  // periods of the same prefix share the first one's counts
    want = j.m[r];
    if (digit > 0) {
      const unsigned long long* pre = w.prefix[(digit - 1) & 1];
      mine = pre[r];
      want = w.want[(digit - 1) & 1][r];
      for (unsigned int q = r; q-- > 0u;)
        if (pre[q] == mine) slot = q;
    } else {
      slot = 0u;
    }
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
      c[q] = w.hist[w.of(digit)][slot][kBins - 1 - (kOwn * u + q)];  // from the top
      sum += c[q];
    }
  }
  unsigned int incl = sum;
#pragma unroll
  for (int dd = 1; dd < 32; dd <<= 1) {
    const unsigned int o = __shfl_up_sync(0xffffffffu, incl, dd);
    if (lane >= static_cast<unsigned int>(dd)) incl += o;
  }
  if (lane == 31u) sm.warp_sum[t >> 5] = incl;
  __syncthreads();
  unsigned long long above = incl - sum;
#pragma unroll
  for (unsigned int q = 0; q < 7; ++q)
    if (q < ((t >> 5) & 7u)) above += sm.warp_sum[r * 8 + q];
  if (live && above < want && want <= above + sum) {
    const int width = digit == 0 ? kBits : wide_shift<kBits>(digit - 1) - wide_shift<kBits>(digit);
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
      if (above < want && want <= above + c[q]) {
        const unsigned long long pre = (mine << width) | (kBins - 1 - (kOwn * u + q)), left = want - above;
        sm.prefix[r] = pre;
        sm.want[r] = left;
        if (blockIdx.x == 0) {
          w.prefix[digit & 1][r] = pre;
          w.want[digit & 1][r] = left;
        }
      }
      above += c[q];
    }
  }
  __syncthreads();
}

template <int kBits>
__global__ void __launch_bounds__(kSelThreads, 1) k_wide_digit(const __grid_constant__ WideBatch b, int digit) {
  __shared__ WideShared<kBits> sm;
  const SelJob& j = b.job[blockIdx.y];
  WideScratch<kBits>& w = static_cast<WideScratch<kBits>*>(b.scratch)[blockIdx.y];
  constexpr int kWords = kSelGroup << kBits;
  const unsigned int t = threadIdx.x;
  for (int i = t; i < kWords; i += kSelThreads) (&sm.hist[0][0])[i] = 0u;
  if (digit > 0) wide_pick<kBits>(j, w, sm, digit - 1);
  if (blockIdx.x == 0)
    for (int i = t; i < kWords; i += kSelThreads) (&w.hist[w.of(digit + 1)][0][0])[i] = 0u;
  __syncthreads();
  // the prefixes counted here: of periods with the same one the first's
  unsigned long long own[kSelGroup];
#pragma unroll
  for (int k = 0; k < kSelGroup; ++k) {
    own[k] = k >= j.g ? ~0ull : digit == 0 ? 0ull : sm.prefix[k];
#pragma unroll
    for (int q = 0; q < k; ++q)
      if (own[q] == own[k]) own[k] = ~0ull;
  }
  const int first = static_cast<int>(blockIdx.x * kSelThreads + t), shift = wide_shift<kBits>(digit);
  constexpr int kStride = kWideCtas * kSelThreads;
  if (shift >= 32) {  // the digit and those before it are in the key's upper half
    unsigned int own32[kSelGroup];
#pragma unroll
    for (int k = 0; k < kSelGroup; ++k) own32[k] = own[k] == ~0ull ? ~0u : static_cast<unsigned int>(own[k]);
    const int sh = shift - 32;
    sel_values<kStride>(j, first, [&](double v, bool valid) {
      const unsigned int h = key_hi(v) >> sh, top = !valid ? ~0u - 1u : digit == 0 ? 0u : h >> kBits;
#pragma unroll
      for (int k = 0; k < kSelGroup; ++k)
        if (top == own32[k]) atomicAdd(&sm.hist[k][h & ((1u << kBits) - 1u)], 1u);
    });
  } else {
    const int width = wide_shift<kBits>(digit - 1) - shift;
    const unsigned int mask = (1u << width) - 1u;
    sel_values<kStride>(j, first, [&](double v, bool valid) {
      const unsigned long long key = key_of(v) >> shift, top = valid ? key >> width : ~0ull - 1ull;
#pragma unroll
      for (int k = 0; k < kSelGroup; ++k)
        if (top == own[k]) atomicAdd(&sm.hist[k][static_cast<unsigned int>(key) & mask], 1u);
    });
  }
  __syncthreads();
  for (int i = t; i < kWords; i += kSelThreads) {
    const unsigned int c = (&sm.hist[0][0])[i];
    if (c) atomicAdd(&(&w.hist[w.of(digit)][0][0])[i], c);
  }
}

template <int kBits>
__global__ void __launch_bounds__(kSelThreads, 1) k_wide_sums(const __grid_constant__ WideBatch b) {
  __shared__ WideShared<kBits> sm;
  __shared__ double part[kSelWarps][kSelGroup];
  __shared__ bool last;
  __shared__ unsigned long long ring[kSelWarps][64];
  const SelJob& j = b.job[blockIdx.y];
  WideScratch<kBits>& w = static_cast<WideScratch<kBits>*>(b.scratch)[blockIdx.y];
  const unsigned int t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  wide_pick<kBits>(j, w, sm, WideScratch<kBits>::kDigits - 1);
  if (blockIdx.x == 0 && static_cast<int>(t) < j.g) {
    if (j.ties) j.ties[t] = sm.want[t];
    j.pml[t] = value_of(sm.prefix[t]);
  }
  if (!j.tvar) return;
  double sum[kSelGroup];
  unsigned long long kth[kSelGroup];
#pragma unroll
  for (int r = 0; r < kSelGroup; ++r) kth[r] = r < j.g ? sm.prefix[r] : ~0ull;
  sel_sums<kWideCtas * kSelThreads>(j, static_cast<int>(blockIdx.x * kSelThreads + t), kth, ring[warp], sum);
#pragma unroll
  for (int r = 0; r < kSelGroup; ++r) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum[r] += __shfl_down_sync(0xffffffffu, sum[r], d);
    if (lane == 0) part[warp][r] = sum[r];
  }
  __syncthreads();
  double* parts = w.parts();
  if (t < static_cast<unsigned int>(kSelGroup)) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < kSelWarps; ++q) s += part[q][t];
    parts[blockIdx.x * kSelGroup + t] = s;
    __threadfence();
  }
  __syncthreads();
  if (t == 0) last = atomicAdd(&w.done, 1u) == static_cast<unsigned int>(kWideCtas - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (static_cast<int>(t) < j.g) {  // the last CTA adds the parts in order
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < kWideCtas; ++c) s += __ldcg(&parts[c * kSelGroup + t]);
    const double v = value_of(sm.prefix[t]);
    j.tvar[t] = (s + static_cast<double>(sm.want[t]) * v) / static_cast<double>(j.m[t]);
  }
}

template <int kBits>
cudaError_t launch_wide_of(const WideBatch& b, int n_jobs, bool sums, cudaStream_t s, int* n_launch) {
  using Scratch = WideScratch<kBits>;
  cudaError_t err = cudaMemsetAsync(b.scratch, 0, sizeof(Scratch) * n_jobs, s);
  if (err != cudaSuccess) return err;
  const dim3 grid(kWideCtas, n_jobs);
  for (int digit = 0; digit < Scratch::kDigits; ++digit) {
    k_wide_digit<kBits><<<grid, kSelThreads, 0, s>>>(b, digit);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  k_wide_sums<kBits><<<sums ? grid : dim3(1, n_jobs), kSelThreads, 0, s>>>(b);
  if (n_launch) *n_launch += Scratch::kDigits + 1;
  return cudaGetLastError();
}

// The widest digits whose scratch fits `bytes` for a job (0: none).
int wide_bits(size_t bytes) {
  return bytes >= sizeof(WideScratch<kWideBits>) ? kWideBits
         : bytes >= sizeof(WideScratch<kWideBitsSmall>) ? kWideBitsSmall
                                                        : 0;
}
cudaError_t launch_wide(const WideBatch& b, int bits, int n_jobs, bool sums, cudaStream_t s, int* n_launch) {
  return bits == kWideBits ? launch_wide_of<kWideBits>(b, n_jobs, sums, s, n_launch)
                           : launch_wide_of<kWideBitsSmall>(b, n_jobs, sums, s, n_launch);
}

// m = ceil(n / rp), within [1, n]
unsigned long long sel_rank(int64_t n, double rp) {
  int64_t m = static_cast<int64_t>(std::ceil(static_cast<double>(n) / rp));
  if (m < 1) m = 1;
  if (m > n) m = n;
  return static_cast<unsigned long long>(m);
}

template <int kCtas>
struct SelLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  SelLaunch(int n_jobs, cudaStream_t s) {
    cfg.gridDim = dim3(kCtas, n_jobs);
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = sizeof(SelShared);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCtas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  SelLaunch(const SelLaunch&) = delete;
  static cudaError_t attributes() {
    const cudaError_t err =
        cudaFuncSetAttribute(k_select<kCtas>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(SelShared));
    return err != cudaSuccess || kCtas <= 8
               ? err
               : cudaFuncSetAttribute(k_select<kCtas>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
};
template <int kCtas>
cudaError_t launch_select_of(const SelBatch& b, int n_jobs, cudaStream_t s) {
  const SelLaunch<kCtas> l(n_jobs, s);
  const cudaError_t err = l.attributes();
  return err != cudaSuccess ? err : cudaLaunchKernelEx(&l.cfg, k_select<kCtas>, b);
}
cudaError_t launch_select(const SelBatch& b, int n_jobs, int ctas, cudaStream_t s) {
  return ctas == 1 ? launch_select_of<1>(b, n_jobs, s)
         : ctas == 4 ? launch_select_of<4>(b, n_jobs, s)
                     : launch_select_of<16>(b, n_jobs, s);
}

// CTAs of a YLT's cluster.  One CTA holds a YLT of up to 8 values a thread; a
// few shorten the passes of a middle one more than their cluster barriers cost.
int sel_ctas(int64_t n) { return n <= 8 * kSelThreads ? 1 : n <= 64 * kSelThreads ? 4 : 16; }

// Whether the current device places a cluster of 16 CTAs (not a portable size:
// a GPC with 16 SMs free for it), asked once a device.
bool sel_places_16() {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];  // 0: not asked, 1: yes, 2: no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return false;
  if (known[dev].load() == 0) {
    SelLaunch<16> l(1, nullptr);
    int clusters = 0;
    const bool ok = l.attributes() == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, k_select<16>, &l.cfg) == cudaSuccess && clusters > 0;
    if (!ok) cudaGetLastError();
    known[dev].store(ok ? 1 : 2);
  }
  return known[dev].load() == 1;
}

// Whether a job takes the wide select: by its YLT's length and its largest
// rank (for k_top_collect's, without sums, 0), so that it gives the same bits in
// any batch.  Above kSelWide the cluster's 16 SMs take longer than all SMs'
// launches, above half of it where a quarter of the values are summed.  Device
// us by cluster and wide, two periods of 100 and 250: 300,000 trials 46 and 79, 1M
// 65 and 80, 2M (4 passes over it) 110 and 88, 16M 860 and 236, 64M 3,420 and
// 686; of 1.05 and 2: 500,000 96 and 83, 1M 163 and 88, 16M 1,870 and 367.  (Five launches with candidates in
// device memory, before the clusters: 1M 95 and 120, 16M 1,000 and 930.)
constexpr int64_t kSelWide = 1 << 20;
bool sel_wide(int64_t n, unsigned long long largest) {
  return n > kSelWide || (n > kSelWide / 2 && largest > static_cast<unsigned long long>(n / 4)) ||
         (sel_ctas(n) == 16 && !sel_places_16());
}
bool sel_may_be_wide(int64_t n) { return sel_wide(n, static_cast<unsigned long long>(n)); }

}  // namespace

size_t select_scratch_bytes(int64_t n, int n_rp) {
  const int groups = (n_rp + kSelGroup - 1) / kSelGroup;
  if (!sel_may_be_wide(n)) return 0;
  return groups < 1 ? sizeof(WideScratch<kWideBitsSmall>)
                    : sizeof(WideScratch<kWideBits>) * static_cast<size_t>(groups < kSelBatchMax ? groups : kSelBatchMax);
}

// A job's periods and ranks, and the largest of these.
static unsigned long long sel_group(const SelectSpec& q, int r0, SelJob* j) {
  j->g = (q.n_rp - r0 < kSelGroup) ? (q.n_rp - r0) : kSelGroup;
  unsigned long long largest = 0ull;
  for (int r = 0; r < kSelGroup; ++r) {
    j->m[r] = r < j->g ? sel_rank(q.n, q.rps[r0 + r]) : 1ull;
    largest = j->m[r] > largest ? j->m[r] : largest;
  }
  return largest;
}

bool select_takes_scratch(const SelectSpec& q) {
  SelJob j;
  for (int r0 = 0; r0 < q.n_rp; r0 += kSelGroup)
    if (sel_wide(q.n, sel_group(q, r0, &j))) return true;
  return false;
}

cudaError_t pml_tvar_batch(const SelectSpec* specs, int n_specs, void* scratch, size_t scratch_bytes, cudaStream_t s,
                           int* n_launch) {
  for (int i = 0; i < n_specs; ++i)
    if (specs[i].n < 1 || specs[i].n_rp < 1) return cudaErrorInvalidValue;
  // one launch (or one of each of the wide select's) per class of lengths and batch of jobs
  WideBatch b;
  b.scratch = scratch;
  const int bits = wide_bits(scratch_bytes);
  const size_t room = bits == kWideBits ? scratch_bytes / sizeof(WideScratch<kWideBits>) : bits ? 1 : 0;
  for (int ctas : {1, 4, 16, kWideCtas}) {
    const bool wide = ctas == kWideCtas;
    const int most = static_cast<int>(wide && room < kSelBatchMax ? room : kSelBatchMax);
    int n_jobs = 0;
    auto flush = [&]() -> cudaError_t {
      if (n_jobs == 0) return cudaSuccess;
      cudaError_t e;
      if (wide) {
        e = launch_wide(b, bits, n_jobs, true, s, n_launch);
      } else {
        SelBatch narrow;
        for (int k = 0; k < n_jobs; ++k) narrow.job[k] = b.job[k];
        e = launch_select(narrow, n_jobs, ctas, s);
        if (n_launch) *n_launch += 1;
      }
      n_jobs = 0;
      return e;
    };
    cudaError_t err;
    for (int i = 0; i < n_specs; ++i) {
      const SelectSpec& q = specs[i];
      for (int r0 = 0; r0 < q.n_rp; r0 += kSelGroup) {
        SelJob j;
        if ((sel_wide(q.n, sel_group(q, r0, &j)) && (room > 0 || !sel_places_16())) != wide || (!wide && sel_ctas(q.n) != ctas))
          continue;
        if (most < 1) return cudaErrorInvalidValue;
        if (n_jobs == most && (err = flush()) != cudaSuccess) return err;
        j.ylt = q.ylt;
        j.n = q.n;
        j.pml = q.pml + r0;
        j.tvar = q.tvar + r0;
        j.ties = nullptr;
        b.job[n_jobs++] = j;
      }
    }
    if ((err = flush()) != cudaSuccess) return err;
  }
  return cudaSuccess;
}

// =============================================================== LSD radix sort
//
// Eight bits a pass, stable.  The items are cut into at most kRxSegments
// segments, one CTA each: k_radix_count counts a segment's digits, and
// k_radix_scatter first sums the segments' counts to its own first places
// (every CTA reads all of them: at most 152 KB, from L2, in place of a scan's
// three launches a pass), then places its items a tile at a time.  An item's
// rank among the tile's equal digits comes from eight ballots a warp (a warp
// match is several times slower) and the warps' counts.  The 16 launches take
// 96 us up to 100,000 year losses, about 6 us each by their latency, and 234 us
// at 1M; with a scan over tiles of 1,024 they were 49 launches, 215 and 356 us.
// Tiles of 2,048: with 4,096 a segment 115 us at 100,000 and no faster at 1M.
// Up to kRxSmall year losses one CTA sorts in shared memory, in one launch: 21
// us at 1,000 and 60 at 8,192, against 116.
namespace {

constexpr int kRxThreads = 512;
constexpr int kRxWarps = kRxThreads / 32;
constexpr int kRxItems = 4;
constexpr int kRxTile = kRxThreads * kRxItems;
constexpr int kRxSegments = 152;  // one CTA an SM
constexpr int kRxSmallThreads = 1024;
constexpr int kRxSmallItems = 8;
constexpr int kRxSmall = kRxSmallThreads * kRxSmallItems;

int radix_segments(int64_t n) {
  const int64_t tiles = (n + kRxTile - 1) / kRxTile;
  return static_cast<int>(tiles < 1 ? 1 : tiles < kRxSegments ? tiles : kRxSegments);
}
// segment s of n_seg: whole tiles
__host__ __device__ __forceinline__ int64_t radix_bound(int64_t n, int n_seg, int s) {
  const int64_t tiles = (n + kRxTile - 1) / kRxTile;
  const int64_t at = tiles * s / n_seg * kRxTile;
  return at < n ? at : n;
}

// The items of a pass: the keys and values of the pass before, or (kYlt) a
// YLT's keys, complemented so that ascending keys are descending losses, and
// their trial indices.
template <bool kYlt>
__device__ __forceinline__ unsigned long long radix_key(const double* ylt, const unsigned long long* keys, int64_t i) {
  if constexpr (kYlt) return ~key_of(ylt[i]);
  else return keys[i];
}

template <bool kYlt>
__global__ void __launch_bounds__(kRxThreads) k_radix_count(const double* ylt, const unsigned long long* keys,
                                                            int64_t n, int shift, unsigned int* counts) {
  __shared__ unsigned int sh[256];
  for (int i = threadIdx.x; i < 256; i += kRxThreads) sh[i] = 0u;
  __syncthreads();
  const int64_t end = radix_bound(n, gridDim.x, blockIdx.x + 1);
#pragma unroll 4
  for (int64_t i = radix_bound(n, gridDim.x, blockIdx.x) + threadIdx.x; i < end; i += kRxThreads)
    atomicAdd(&sh[(radix_key<kYlt>(ylt, keys, i) >> shift) & 255u], 1u);
  __syncthreads();
  if (threadIdx.x < 256) counts[blockIdx.x * 256 + threadIdx.x] = sh[threadIdx.x];
}

// The lanes whose digit is this lane's, among the valid ones.
__device__ __forceinline__ unsigned int radix_peers(unsigned int d, bool valid) {
  unsigned int peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned int b = __ballot_sync(0xffffffffu, (d >> k) & 1u);
    peers &= ((d >> k) & 1u) ? b : ~b;
  }
  return peers;
}

template <bool kYlt, class V, class VOut>
__global__ void __launch_bounds__(kRxThreads) k_radix_scatter(const double* ylt, const unsigned long long* keys,
                                                              const V* vals, int64_t n, int shift,
                                                              const unsigned int* counts,
                                                              unsigned long long* keys_out, VOut* vals_out) {
  __shared__ unsigned int wc[kRxWarps][256];  // per warp: a digit's count in the tile, then the place of its items
  __shared__ unsigned int base[256];          // the segment's next place of each digit
  __shared__ unsigned int part[2][kRxThreads];
  __shared__ unsigned int warp_sum[8];
  const unsigned int t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  {
    // the segments before this one and all segments, a digit a thread over a part of the segments
    constexpr unsigned int kParts = kRxThreads / 256;
    const unsigned int d = t & 255u;
    unsigned int before = 0u, total = 0u;
#pragma unroll 8
    for (unsigned int s = t >> 8; s < gridDim.x; s += kParts) {
      const unsigned int c = counts[s * 256 + d];
      total += c;
      before += s < blockIdx.x ? c : 0u;
    }
    part[0][t] = before;
    part[1][t] = total;
    __syncthreads();
    unsigned int incl = 0u;
    if (t < 256u) {
#pragma unroll
      for (unsigned int q = 1; q < kParts; ++q) {
        before += part[0][q * 256 + t];
        total += part[1][q * 256 + t];
      }
      incl = total;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        const unsigned int o = __shfl_up_sync(0xffffffffu, incl, dd);
        if (lane >= static_cast<unsigned int>(dd)) incl += o;
      }
      if (lane == 31u) warp_sum[warp] = incl;
    }
    __syncthreads();
    if (t < 256u) {
      unsigned int at = incl - total + before;
      for (unsigned int w = 0; w < warp; ++w) at += warp_sum[w];
      base[t] = at;
    }
  }
  const int64_t end = radix_bound(n, gridDim.x, blockIdx.x + 1);
  for (int64_t tile = radix_bound(n, gridDim.x, blockIdx.x); tile < end; tile += kRxTile) {
    __syncthreads();  // the tile before is placed (and base is there)
    for (int i = lane; i < 256; i += 32) wc[warp][i] = 0u;
    __syncwarp();
    unsigned long long key[kRxItems];
    V val[kRxItems];
    unsigned int at[kRxItems];
#pragma unroll
    for (int j = 0; j < kRxItems; ++j) {
      const int64_t i = tile + warp * (32 * kRxItems) + 32 * j + lane;
      key[j] = i < end ? radix_key<kYlt>(ylt, keys, i) : 0ull;
      if constexpr (kYlt) val[j] = static_cast<V>(i);
      else val[j] = i < end ? vals[i] : V{};
    }
#pragma unroll
    for (int j = 0; j < kRxItems; ++j) {
      const bool valid = tile + warp * (32 * kRxItems) + 32 * j + lane < end;
      const unsigned int d = static_cast<unsigned int>(key[j] >> shift) & 255u;
      const unsigned int peers = radix_peers(d, valid);
      const unsigned int below = __popc(peers & ((1u << lane) - 1u));
      const unsigned int have = wc[warp][d];
      __syncwarp();
      if (valid && below == 0u) wc[warp][d] = have + __popc(peers);
      __syncwarp();
      at[j] = have + below;
    }
    __syncthreads();
    if (t < 256u) {
      unsigned int run = base[t];
#pragma unroll
      for (int w = 0; w < kRxWarps; ++w) {
        const unsigned int c = wc[w][t];
        wc[w][t] = run;
        run += c;
      }
      base[t] = run;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRxItems; ++j)
      if (tile + warp * (32 * kRxItems) + 32 * j + lane < end) {
        const unsigned int dst = at[j] + wc[warp][(key[j] >> shift) & 255u];
        if (keys_out) keys_out[dst] = key[j];
        vals_out[dst] = static_cast<VOut>(val[j]);
      }
  }
}

struct RxSmall {
  unsigned long long key[kRxSmall];
  uint32_t val[kRxSmall];
  unsigned int wc[kRxSmallThreads / 32][256];
  unsigned int first[256];
  unsigned int warp_sum[8];
};

// The order of at most kRxSmall items, all passes in one CTA.
template <bool kYlt>
__global__ void __launch_bounds__(kRxSmallThreads, 1) k_radix_small(const double* ylt,
                                                                        const unsigned long long* keys,
                                                                        const uint32_t* vals, int n, int64_t* order) {
  extern __shared__ __align__(16) unsigned char rx_smem[];
  RxSmall& sm = *reinterpret_cast<RxSmall*>(rx_smem);
  const unsigned int t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  // the warps that hold items; a warp's items are contiguous
  const int per_warp = 32 * kRxSmallItems, i0 = static_cast<int>(warp) * per_warp + static_cast<int>(lane);
  const unsigned int n_warps = static_cast<unsigned int>((n + per_warp - 1) / per_warp);
  unsigned long long key[kRxSmallItems];
  uint32_t val[kRxSmallItems];
#pragma unroll
  for (int j = 0; j < kRxSmallItems; ++j) {
    key[j] = i0 + 32 * j < n ? radix_key<kYlt>(ylt, keys, i0 + 32 * j) : 0ull;
    val[j] = kYlt ? static_cast<uint32_t>(i0 + 32 * j) : i0 + 32 * j < n ? vals[i0 + 32 * j] : 0u;
  }
#pragma unroll 1
  for (int shift = 0; shift < 64; shift += 8) {
    unsigned int at[kRxSmallItems];
    for (int i = lane; i < 256; i += 32) sm.wc[warp][i] = 0u;
    __syncwarp();
    if (warp < n_warps) {
#pragma unroll
      for (int j = 0; j < kRxSmallItems; ++j) {
        const bool valid = i0 + 32 * j < n;
        const unsigned int d = static_cast<unsigned int>(key[j] >> shift) & 255u;
        const unsigned int peers = radix_peers(d, valid);
        const unsigned int below = __popc(peers & ((1u << lane) - 1u));
        const unsigned int have = sm.wc[warp][d];
        __syncwarp();
        if (valid && below == 0u) sm.wc[warp][d] = have + __popc(peers);
        __syncwarp();
        at[j] = have + below;
      }
    }
    __syncthreads();
    unsigned int total = 0u, incl = 0u;
    if (t < 256u) {
#pragma unroll 8
      for (unsigned int w = 0; w < kRxSmallThreads / 32; ++w) {
        const unsigned int c = sm.wc[w][t];
        sm.wc[w][t] = total;
        total += c;
      }
      incl = total;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        const unsigned int o = __shfl_up_sync(0xffffffffu, incl, dd);
        if (lane >= static_cast<unsigned int>(dd)) incl += o;
      }
      if (lane == 31u) sm.warp_sum[warp] = incl;
    }
    __syncthreads();
    if (t < 256u) {
      unsigned int first = incl - total;
      for (unsigned int w = 0; w < warp; ++w) first += sm.warp_sum[w];
      sm.first[t] = first;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRxSmallItems; ++j)
      if (i0 + 32 * j < n) {
        const unsigned int d = static_cast<unsigned int>(key[j] >> shift) & 255u;
        const unsigned int dst = at[j] + sm.wc[warp][d] + sm.first[d];
        sm.key[dst] = key[j];
        sm.val[dst] = val[j];
      }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRxSmallItems; ++j)
      if (i0 + 32 * j < n) {
        key[j] = sm.key[i0 + 32 * j];
        val[j] = sm.val[i0 + 32 * j];
      }
  }
#pragma unroll
  for (int j = 0; j < kRxSmallItems; ++j)
    if (i0 + 32 * j < n) order[i0 + 32 * j] = static_cast<int64_t>(val[j]);
}

}  // namespace

namespace {

// scratch of the passes: two key and two index arrays, then the segments' digit counts
struct RxScratch {
  unsigned long long* keys[2];
  uint32_t* vals[2];
  unsigned int* counts;
};
size_t radix_scratch_bytes(int64_t n) {
  return static_cast<size_t>(n) * 2 * (sizeof(unsigned long long) + sizeof(uint32_t)) +
         sizeof(unsigned int) * 256 * static_cast<size_t>(radix_segments(n)) + 256;
}
RxScratch radix_scratch(void* scratch, int64_t n) {
  RxScratch x;
  x.keys[0] = static_cast<unsigned long long*>(scratch);
  x.keys[1] = x.keys[0] + n;
  x.vals[0] = reinterpret_cast<uint32_t*>(x.keys[1] + n);
  x.vals[1] = x.vals[0] + n;
  x.counts = reinterpret_cast<unsigned int*>(x.vals[1] + n);
  return x;
}

// The indices in ascending key order: of a YLT (kYlt), or of n (key, index)
// pairs in x.keys[1] and x.vals[1].
template <bool kYlt>
cudaError_t radix_order(const double* ylt, const RxScratch& x, int64_t n, int64_t* order, cudaStream_t s,
                        int* n_launch) {
  cudaError_t err;
  if (n <= kRxSmall) {
    if ((err = cudaFuncSetAttribute(k_radix_small<kYlt>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    sizeof(RxSmall))) != cudaSuccess)
      return err;
    k_radix_small<kYlt><<<1, kRxSmallThreads, sizeof(RxSmall), s>>>(ylt, x.keys[1], x.vals[1], static_cast<int>(n),
                                                                   order);
    if (n_launch) *n_launch += 1;
    return cudaGetLastError();
  }
  const int n_seg = radix_segments(n);
  for (int pass = 0; pass < 8; ++pass) {
    const int shift = 8 * pass, from = (pass + 1) & 1, to = pass & 1;
    if (kYlt && pass == 0) {
      k_radix_count<true><<<n_seg, kRxThreads, 0, s>>>(ylt, nullptr, n, shift, x.counts);
      k_radix_scatter<true, uint32_t, uint32_t><<<n_seg, kRxThreads, 0, s>>>(ylt, nullptr, nullptr, n, shift, x.counts,
                                                                            x.keys[to], x.vals[to]);
    } else {
      k_radix_count<false><<<n_seg, kRxThreads, 0, s>>>(nullptr, x.keys[from], n, shift, x.counts);
      if (pass < 7)
        k_radix_scatter<false, uint32_t, uint32_t><<<n_seg, kRxThreads, 0, s>>>(
            nullptr, x.keys[from], x.vals[from], n, shift, x.counts, x.keys[to], x.vals[to]);
      else
        k_radix_scatter<false, uint32_t, int64_t><<<n_seg, kRxThreads, 0, s>>>(
            nullptr, x.keys[from], x.vals[from], n, shift, x.counts, nullptr, order);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  if (n_launch) *n_launch += 16;
  return cudaSuccess;
}

}  // namespace

size_t sort_scratch_bytes(int64_t n) { return radix_scratch_bytes(n); }

cudaError_t sort_desc_device(const double* ylt, int64_t n, int64_t* order, void* scratch, cudaStream_t s,
                             int* n_launch) {
  return radix_order<true>(ylt, radix_scratch(scratch, n), n, order, s, n_launch);
}

size_t sort_pairs_scratch_bytes(int64_t n) {
  return static_cast<size_t>(n) * (sizeof(unsigned long long) + sizeof(int64_t)) +
         sizeof(unsigned int) * 256 * static_cast<size_t>(radix_segments(n)) + 256;
}

cudaError_t sort_pairs_ascending(unsigned long long* keys, int64_t* vals, int64_t n, int key_bits, void* scratch,
                                 cudaStream_t s, int* n_launch) {
  const int passes = (key_bits + 7) / 8;
  const int n_seg = radix_segments(n);
  unsigned long long* keys_b = static_cast<unsigned long long*>(scratch);
  int64_t* vals_b = reinterpret_cast<int64_t*>(keys_b + n);
  unsigned int* counts = reinterpret_cast<unsigned int*>(vals_b + n);
  cudaError_t err = cudaSuccess;
  // an odd number of passes ends in the scratch buffers: the data start there, so the result
  // lands in (keys, vals)
  unsigned long long *ki = keys, *ko = keys_b;
  int64_t *ii = vals, *io = vals_b;
  if (passes & 1) {
    if ((err = cudaMemcpyAsync(keys_b, keys, sizeof(unsigned long long) * n, cudaMemcpyDeviceToDevice, s)) ||
        (err = cudaMemcpyAsync(vals_b, vals, sizeof(int64_t) * n, cudaMemcpyDeviceToDevice, s)))
      return err;
    ki = keys_b;
    ko = keys;
    ii = vals_b;
    io = vals;
  }
  for (int pass = 0; pass < passes; ++pass) {
    k_radix_count<false><<<n_seg, kRxThreads, 0, s>>>(nullptr, ki, n, 8 * pass, counts);
    k_radix_scatter<false, int64_t, int64_t><<<n_seg, kRxThreads, 0, s>>>(nullptr, ki, ii, n, 8 * pass, counts, ko,
                                                                         io);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    std::swap(ki, ko);
    std::swap(ii, io);
  }
  if (n_launch) *n_launch += 2 * passes;
  return cudaSuccess;
}

namespace {

// The first m_valid entries of a descending order: values and global trial
// indices (trial_offset + local index); entries m_valid..m-1 are padding
// (-inf, -1).
__global__ void k_top_gather(const double* ylt, const int64_t* order, int64_t m_valid, int64_t m,
                             int64_t trial_offset, double* vals, int64_t* trials) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < m; i += stride) {
    if (i < m_valid) {
      const int64_t t = order[i];
      vals[i] = ylt[t];
      trials[i] = trial_offset + t;
    } else {
      vals[i] = -__longlong_as_double(0x7FF0000000000000ll);
      trials[i] = -1;
    }
  }
}

// The m largest without the whole order: the m-th key comes from k_select, and
// these kernels collect, in trial order, the values above it and the first of
// its ties (as many as the m largest hold).  Segment s of the YLT is a CTA's;
// counts[2 s] and [2 s + 1]: its values above the m-th key and its ties.
constexpr int kTopThreads = 1024;
constexpr int kTopSegments = 152;

struct TopKth {
  double value;            // the m-th largest value
  unsigned long long ties;  // of its ties, how many are among the m largest
};

__global__ void __launch_bounds__(kTopThreads) k_top_count(const double* ylt, int64_t n, const TopKth* kth,
                                                           unsigned int* counts) {
  __shared__ unsigned int s_above, s_ties;
  if (threadIdx.x == 0) s_above = s_ties = 0u;
  __syncthreads();
  const unsigned long long k = key_of(kth->value);
  const int64_t begin = n * blockIdx.x / gridDim.x, end = n * (blockIdx.x + 1) / gridDim.x;
  unsigned int above = 0u, ties = 0u;
#pragma unroll 4
  for (int64_t i = begin + threadIdx.x; i < end; i += kTopThreads) {
    const unsigned long long x = key_of(ylt[i]);
    above += x > k;
    ties += x == k;
  }
  above = __reduce_add_sync(0xffffffffu, above);
  ties = __reduce_add_sync(0xffffffffu, ties);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_above, above);
    atomicAdd(&s_ties, ties);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    counts[2 * blockIdx.x] = s_above;
    counts[2 * blockIdx.x + 1] = s_ties;
  }
}

__global__ void __launch_bounds__(kTopThreads) k_top_collect(const double* ylt, int64_t n, const TopKth* kth,
                                                             const unsigned int* counts, unsigned long long* keys,
                                                             uint32_t* idx) {
  __shared__ unsigned int w_above[kTopThreads / 32], w_ties[kTopThreads / 32];
  const unsigned int t = threadIdx.x, lane = t & 31u, warp = t >> 5, lt = (1u << lane) - 1u;
  const unsigned long long k = key_of(kth->value), most = kth->ties;
  // the items before this segment
  unsigned long long above = 0ull, ties = 0ull;
  for (unsigned int s = 0; s < blockIdx.x; ++s) {
    above += counts[2 * s];
    ties += counts[2 * s + 1];
  }
  const int64_t begin = n * blockIdx.x / gridDim.x, end = n * (blockIdx.x + 1) / gridDim.x;
  for (int64_t i0 = begin; i0 < end; i0 += kTopThreads) {
    const int64_t i = i0 + t;
    const unsigned long long x = i < end ? key_of(ylt[i]) : 0ull;
    const unsigned int a = __ballot_sync(0xffffffffu, i < end && x > k), e = __ballot_sync(0xffffffffu, i < end && x == k);
    if (lane == 0) {
      w_above[warp] = __popc(a);
      w_ties[warp] = __popc(e);
    }
    __syncthreads();
    unsigned int pa = lane < warp ? w_above[lane] : 0u, pe = lane < warp ? w_ties[lane] : 0u;
    unsigned int ta = w_above[lane], te = w_ties[lane];
    pa = __reduce_add_sync(0xffffffffu, pa);
    pe = __reduce_add_sync(0xffffffffu, pe);
    ta = __reduce_add_sync(0xffffffffu, ta);
    te = __reduce_add_sync(0xffffffffu, te);
    const unsigned long long my_ties = ties + pe + __popc(e & lt);  // ties before this item
    const unsigned long long at = above + pa + __popc(a & lt) + (my_ties < most ? my_ties : most);
    if (i < end && (x > k || (x == k && my_ties < most))) {
      keys[at] = ~x;
      idx[at] = static_cast<uint32_t>(i);
    }
    above += ta;
    ties += te;
    __syncthreads();
  }
}

}  // namespace

cudaError_t top_gather_device(const double* ylt, const int64_t* order, int64_t m_valid, int64_t m, int64_t trial_offset,
                              double* vals, int64_t* trials, cudaStream_t s) {
  const int64_t blocks = (m + 255) / 256;
  k_top_gather<<<static_cast<int>(blocks < 1024 ? (blocks > 0 ? blocks : 1) : 1024), 256, 0, s>>>(
      ylt, order, m_valid, m, trial_offset, vals, trials);
  return cudaGetLastError();
}

// scratch: the m-th value, the segments' counts, the wide select's, the sort's
constexpr size_t kTopCountsBytes = (2 * sizeof(unsigned int) * kTopSegments + 255) & ~size_t(255);
constexpr size_t kTopWideBytes = (sizeof(WideScratch<kWideBits>) + 255) & ~size_t(255);

size_t top_wide_bytes(int64_t n) { return sel_wide(n, 0) ? kTopWideBytes : 0; }

size_t top_scratch_bytes(int64_t n, int64_t m) {
  return radix_scratch_bytes(m) + 256 + kTopCountsBytes + top_wide_bytes(n);
}

cudaError_t top_order_device(const double* ylt, int64_t n, int64_t m, int64_t* order, void* scratch, cudaStream_t s,
                             int* n_launch) {
  unsigned char* base = static_cast<unsigned char*>(scratch);
  TopKth* kth = reinterpret_cast<TopKth*>(base);
  unsigned int* counts = reinterpret_cast<unsigned int*>(base + 256);
  const RxScratch x = radix_scratch(base + 256 + kTopCountsBytes + top_wide_bytes(n), m);
  SelJob j;
  j.ylt = ylt;
  j.n = n;
  j.pml = &kth->value;
  j.tvar = nullptr;
  j.ties = &kth->ties;
  j.g = 1;
  for (int r = 0; r < kSelGroup; ++r) j.m[r] = r == 0 ? static_cast<unsigned long long>(m) : 1ull;
  cudaError_t err;
  if (sel_wide(n, 0)) {
    WideBatch b;
    b.job[0] = j;
    b.scratch = base + 256 + kTopCountsBytes;
    err = launch_wide(b, kWideBits, 1, false, s, n_launch);
  } else {
    SelBatch b;
    b.job[0] = j;
    err = launch_select(b, 1, sel_ctas(n), s);
    if (n_launch) *n_launch += 1;
  }
  if (err != cudaSuccess) return err;
  k_top_count<<<kTopSegments, kTopThreads, 0, s>>>(ylt, n, kth, counts);
  k_top_collect<<<kTopSegments, kTopThreads, 0, s>>>(ylt, n, kth, counts, x.keys[1], x.vals[1]);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  if (n_launch) *n_launch += 2;
  return radix_order<false>(nullptr, x, m, order, s, n_launch);
}

}  // namespace ara

// =============================================================== allocation-free PML / TVaR
//
// A fixed block of device memory, owned by the library, holds the device
// outputs of ara_pml_tvar_noalloc for host arrays and the wide select's scratch
// (the other selects' state is in shared memory).  In host code the name of a __device__ array is only a host-side stand-in; the kernels get
// the block's device address, looked up once per device.
namespace {

static __device__ __align__(256) unsigned char g_noalloc_scratch[ARA_NOALLOC_SCRATCH_BYTES];

constexpr int kNoallocMaxDevices = 64;
void* g_noalloc_addr[kNoallocMaxDevices] = {};  // device address of the block, per device

constexpr size_t kNoallocOutBytes = 2 * ARA_NOALLOC_MAX_RP * sizeof(double);
static_assert(ARA_NOALLOC_SCRATCH_BYTES >= kNoallocOutBytes + sizeof(ara::WideScratch<ara::kWideBitsSmall>) && kNoallocOutBytes % 16 == 0,
              "fixed block too small for the outputs and a job's scratch");

}  // namespace

extern "C" ARA_API int ara_pml_tvar_noalloc(const double* ylt, int64_t n, const double* return_periods, int32_t n_rp,
                                            double* pml_out, double* tvar_out, void* cuda_stream) {
  if (!ylt || n < 1 || !return_periods || n_rp < 1 || n_rp > ARA_NOALLOC_MAX_RP || !pml_out || !tvar_out)
    return ARA_EINVAL;
  for (int32_t r = 0; r < n_rp; ++r)
    if (!(return_periods[r] >= 1.0) || !std::isfinite(return_periods[r])) return ARA_EINVAL;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, ylt) != cudaSuccess) {
    cudaGetLastError();
    return ARA_EINVAL;
  }
  if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) return ARA_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return ARA_ECUDA;
  // memory of another GPU would be read as a peer access
  if (at.type == cudaMemoryTypeDevice && at.device != dev) return ARA_EINVAL;
  // set-up, once per device (with that device current): the block's device address
  if (g_noalloc_addr[dev] == nullptr) {
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || addr == nullptr) {
      cudaGetLastError();
      return ARA_ECUDA;
    }
    g_noalloc_addr[dev] = addr;
  }
  unsigned char* block = static_cast<unsigned char*>(g_noalloc_addr[dev]);
  double* d_out = reinterpret_cast<double*>(block);  // 2 * ARA_NOALLOC_MAX_RP doubles, then a wide select's scratch
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // 0: host memory, 1: device (or managed) memory of this GPU, -1: another GPU's memory
  auto kind_of = [dev](const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    if (a.type == cudaMemoryTypeManaged) return 1;
    if (a.type == cudaMemoryTypeDevice) return a.device == dev ? 1 : -1;
    return 0;
  };
  const int pml_kind = kind_of(pml_out), tvar_kind = kind_of(tvar_out);
  if (pml_kind < 0 || tvar_kind < 0) return ARA_EINVAL;
  const bool pml_dev = pml_kind == 1, tvar_dev = tvar_kind == 1;
  double* d_pml = pml_dev ? pml_out : d_out;
  double* d_tvar = tvar_dev ? tvar_out : d_out + ARA_NOALLOC_MAX_RP;
  const ara::SelectSpec spec{ylt, n, return_periods, n_rp, d_pml, d_tvar};
  if (ara::pml_tvar_batch(&spec, 1, block + kNoallocOutBytes, ARA_NOALLOC_SCRATCH_BYTES - kNoallocOutBytes, s,
                          nullptr) != cudaSuccess)
    return ARA_ECUDA;
  if (!pml_dev && cudaMemcpyAsync(pml_out, d_pml, sizeof(double) * n_rp, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return ARA_ECUDA;
  if (!tvar_dev && cudaMemcpyAsync(tvar_out, d_tvar, sizeof(double) * n_rp, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return ARA_ECUDA;
  if ((!pml_dev || !tvar_dev) && cudaStreamSynchronize(s) != cudaSuccess) return ARA_ECUDA;
  return ARA_OK;
}
