// Exclusive prefix sums of uint64 arrays (bit offsets o_i of Sec. 6.3), in one
// launch.
#include "lookback.cuh"

namespace rs {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr uint64_t kTile = uint64_t(kThreads) * kItems;

__global__ void __launch_bounds__(kThreads) k_scan(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                   uint64_t count, LookState st, int* error) {
  __shared__ uint32_t tile_s;
  __shared__ uint64_t before_s;
  if (threadIdx.x == 0) tile_s = atomicAdd(st.ticket, 1u);
  __syncthreads();
  const uint32_t tile = tile_s;
  const uint64_t base = tile * kTile + threadIdx.x * uint64_t(kItems);
  uint64_t v[kItems], s[1] = {0}, run[1], total[1];
#pragma unroll
  for (int k = 0; k < kItems; k++) {
    v[k] = base + k < count ? in[base + k] : 0;
    s[0] += v[k];
  }
  block_scan<1, kThreads>(s, run, total);
  if (threadIdx.x < 32) {
    uint64_t before[1];
    look_back<1>(st, tile, total, before, error);
    if (threadIdx.x == 0) before_s = before[0];
  }
  __syncthreads();
  uint64_t at = run[0] + before_s;
#pragma unroll
  for (int k = 0; k < kItems; k++) {
    if (base + k < count) out[base + k] = at;
    at += v[k];
  }
  if (threadIdx.x == kThreads - 1 && (tile + 1) * kTile >= count) out[count] = at;
}

}  // namespace

uint64_t scan_tiles(uint64_t count) { return (count + kTile - 1) / kTile; }

int exclusive_scan_u64(const uint64_t* in, uint64_t* out, uint64_t count, const LookState& st, int* error,
                       cudaStream_t s) {
  if (count == 0) {
    RS_CUDA(cudaMemsetAsync(out, 0, sizeof(uint64_t), s));
    return RECSPLIT_OK;
  }
  k_scan<<<static_cast<unsigned>(scan_tiles(count)), kThreads, 0, s>>>(in, out, count, st, error);
  count_launch();
  RS_CUDA(cudaGetLastError());
  return RECSPLIT_OK;
}

}  // namespace rs
