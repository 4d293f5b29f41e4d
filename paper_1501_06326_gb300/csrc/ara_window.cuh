// Windows of (event, ELT) pairs: how the losses kernels give the lanes of a
// warp the pairs of the next hit events.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ara {

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// A window: up to 32 pairs of whole events, one per lane.  Of lane q < np: its
// event's record (x, y), the event's first lane and its place among the
// window's events; of lane i < n_take: its own event's first lane.
struct PairWindow {
  uint32_t ex, ey, epre, ev, np, pre;
  int n_take;  // events
};

// The window of the first events of lanes' records (cnt: lane's event's pairs, 0 beyond the last).
__device__ __forceinline__ PairWindow make_window(uint2 r, uint32_t cnt) {
  const uint32_t q = threadIdx.x & 31;
  PairWindow w;
  const uint32_t incl = warp_inclusive_scan(cnt);
  const uint32_t pre = w.pre = incl - cnt;
  const bool take = cnt != 0 && incl <= 32u;
  w.n_take = __popc(__ballot_sync(0xffffffffu, take));
  w.np = w.n_take > 0 ? __shfl_sync(0xffffffffu, incl, w.n_take - 1) : 0u;
  const uint32_t starts = __reduce_or_sync(0xffffffffu, take ? (1u << pre) : 0u);
  // lane q's event: the last start at or below q
  w.ev = static_cast<uint32_t>(__popc(starts & (0xffffffffu >> (31u - q)))) - 1u;
  w.ex = __shfl_sync(0xffffffffu, r.x, w.ev);
  w.ey = __shfl_sync(0xffffffffu, r.y, w.ev);
  w.epre = __shfl_sync(0xffffffffu, pre, w.ev);
  return w;
}

}  // namespace ara
