// Exclusive prefix of a tile in a one-launch scan: every tile publishes its
// sums, then looks back over its predecessors' until it meets one whose prefix
// is complete (Merrill and Garland, "Single-pass Parallel Prefix Scan with
// Decoupled Look-back", 2016).  Tiles take their numbers from a counter in the
// order they start, so the tiles a tile waits for are running or done.
#pragma once

#include "common.h"

namespace rs {

// A scan in three launches (tile sums, their scan, the tiles) cost 13 us for
// 2 * 10^4 values, three times in a build; in one launch it takes 4.
constexpr uint32_t kLookSpin = 1u << 22;  // polls of one predecessor before giving up

// State of a scan of N values a tile: flag (0 nothing, 1 sums, 2 prefix; zero
// before the launch), sums and inclusive prefixes, N words per tile each.
struct LookState {
  uint32_t* flag;
  uint64_t* sums;
  uint64_t* prefix;
  uint32_t* ticket;  // zero before the launch
};

// Called by a whole warp with the tile's sums in every lane: the exclusive
// prefix of the tile, in every lane.  After kLookSpin polls without an answer
// *error is set and the prefix is 0 (the values stay below the scan's total).
template <int N>
__device__ __forceinline__ void look_back(const LookState& st, uint32_t tile, const uint64_t (&sum)[N],
                                          uint64_t (&before)[N], int* error) {
  const uint32_t lane = threadIdx.x & 31;
  volatile uint32_t* flag = st.flag;
#pragma unroll
  for (int k = 0; k < N; k++) before[k] = 0;
  if (tile) {
    if (lane < N) st.sums[uint64_t(tile) * N + lane] = sum[lane];
    __threadfence();
    __syncwarp();
    if (lane == 0) flag[tile] = 1;
    for (uint32_t end = tile;;) {  // predecessors end - 1, end - 2, ...: one per lane
      uint32_t f = 2;
      const bool some = lane < end;
      const uint32_t p = some ? end - 1 - lane : 0;
      if (some) {
        uint32_t polls = 0;
        while ((f = flag[p]) == 0 && ++polls < kLookSpin) {
        }
      }
      __threadfence();
      if (__any_sync(0xFFFFFFFFu, f == 0)) {
        if (lane == 0) atomicCAS(error, 0, RECSPLIT_E_INVALID);
#pragma unroll
        for (int k = 0; k < N; k++) before[k] = 0;
        break;
      }
      const uint32_t done = __ballot_sync(0xFFFFFFFFu, f == 2);  // lanes beyond the first tile count as done, with 0
      const uint32_t last = done ? __ffs(done) - 1 : 31;
#pragma unroll
      for (int k = 0; k < N; k++) {
        uint64_t v = 0;
        if (some && lane <= last)
          v = *reinterpret_cast<volatile uint64_t*>((f == 2 ? st.prefix : st.sums) + uint64_t(p) * N + k);
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        before[k] += v;
      }
      if (done) break;
      end -= 32;
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < N; k++) st.prefix[uint64_t(tile) * N + k] = before[k] + sum[k];
    __threadfence();
    flag[tile] = 2;
  }
}

// Exclusive scan over the CTA (THREADS threads) of N values a thread, and the
// CTA's sums.
template <int N, int THREADS>
__device__ __forceinline__ void block_scan(const uint64_t (&v)[N], uint64_t (&before)[N], uint64_t (&total)[N]) {
  __shared__ uint64_t warp_sums[N][THREADS / 32];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t x[N];
#pragma unroll
  for (int k = 0; k < N; k++) {
    x[k] = v[k];
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x[k], o);
      if (lane >= o) x[k] += y;
    }
    if (lane == 31) warp_sums[k][warp] = x[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; k++) {
    uint64_t s = 0, all = 0;
#pragma unroll
    for (uint32_t w = 0; w < THREADS / 32; w++) {
      const uint64_t y = warp_sums[k][w];
      s += w < warp ? y : 0;
      all += y;
    }
    before[k] = s + x[k] - v[k];
    total[k] = all;
  }
  __syncthreads();
}

}  // namespace rs
