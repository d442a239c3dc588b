// Construction of one or many structures in one pass: signatures and buckets
// (Sec. 6.1), grouping by bucket (Sec. 9), the level-by-level searches
// (search.cu), Golomb-Rice encoding (Sec. 6.2) and the double Elias-Fano lists
// (Sec. 6.3, Sec. 7.4).
//
// A batch is a list of key sets with their own leaf and bucket sizes.  All
// keys, buckets and tree nodes of all sets share the device arrays (indices
// are global; per-set bases map them back), so one launch of each kernel
// covers every set: one signature pass, one scan, one queue of split nodes
// per tree level, one leaf launch per distinct leaf size.  Nodes carry the
// parameter class of their set.  A single build is a batch of one.
//
// Host synchronisations: one after the bucket histogram (largest bucket per
// leaf size -> tables and level plan) and one after the bit lengths (tree
// size and Elias-Fano parameters per set -> layout of the structures).  With
// BuildOptions::use_graph the searches and the length computation between
// them are captured in a CUDA graph and launched as one.
#include <algorithm>
#include <climits>
#include <cstring>
#include <map>

#include <nvtx3/nvToolsExt.h>

#include "device.cuh"
#include "lookback.cuh"

namespace rs {

DeviceMem::~DeviceMem() {
  if (p) cudaFreeAsync(p, nullptr);
}

namespace {

constexpr int kBlock = 256;
constexpr int kTileItems = 8;
constexpr uint64_t kTile = uint64_t(kBlock) * kTileItems;  // keys, buckets or elements per block

inline unsigned grid_for(uint64_t n, int block = kBlock) {
  uint64_t g = (n + block - 1) / block;
  return static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>(g, 1u << 30)));
}

// Per-set description on the device.
struct DevSet {
  const uint64_t* u64;
  const uint8_t* bytes;
  const uint64_t* offsets;
  uint64_t n, key_base, nb, bucket_base;
  uint32_t cls, leaf;
  uint64_t key_tile_base, bucket_tile_base, elem_tile_base;  // first block of the set in each tiling
  uint64_t lane_base;     // first lane of the set in the kernels over codes (bucket_lane)
  uint32_t warp_buckets;  // a warp per bucket there, else a lane
};

// Set whose tile range contains block `blk` (tile bases are non-decreasing).
__device__ __forceinline__ uint32_t set_of_block(const DevSet* sets, uint32_t count, uint64_t blk, int which) {
  uint32_t lo = 0, hi = count;  // first set with base > blk, minus one
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    const uint64_t b = which == 0 ? sets[mid].key_tile_base
                                  : (which == 1 ? sets[mid].bucket_tile_base : sets[mid].elem_tile_base);
    if (b <= blk)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo - 1;
}

// ---------------------------------------------------------------- A1/A2
// Signature of every key, its global bucket, and the bucket histogram.
// A byte-string key with start > end or end > offsets[n] (offsets must not
// decrease) is read as the empty string and flags *bad_offsets: the build
// then fails with RECSPLIT_E_INVALID, and no read leaves bytes[0 .. offsets[n]),
// the span the caller provides.
__global__ void __launch_bounds__(kBlock) k_signature(const DevSet* __restrict__ sets, uint32_t count,
                                                      uint32_t* __restrict__ bucket, uint64_t* __restrict__ lo,
                                                      unsigned long long* __restrict__ counts,
                                                      int* __restrict__ bad_offsets) {
  const uint32_t si = set_of_block(sets, count, blockIdx.x, 0);
  const DevSet st = sets[si];
  const uint64_t t0 = (blockIdx.x - st.key_tile_base) * kTile;
#pragma unroll 2
  for (int k = 0; k < kTileItems; k++) {
    const uint64_t j = t0 + uint64_t(k) * kBlock + threadIdx.x;
    if (j >= st.n) break;
    uint64_t h, l;
    if (st.u64) {
      signature_u64(__ldg(st.u64 + j), h, l);
    } else {
      const uint64_t o0 = __ldg(st.offsets + j), o1 = __ldg(st.offsets + j + 1);
      const bool ok = o0 <= o1 && o1 <= __ldg(st.offsets + st.n);
      if (!ok) *bad_offsets = 1;
      signature_bytes(st.bytes + (ok ? o0 : 0), ok ? o1 - o0 : 0, h, l);
    }
    const uint64_t b = st.bucket_base + bucket_of(h, st.nb);
    const uint64_t i = st.key_base + j;
    bucket[i] = static_cast<uint32_t>(b);
    lo[i] = l;
    atomicAdd(counts + b, 1ull);
  }
}

// Per bucket: its set, and the per-class largest / per-set smallest bucket
// (the smallest as the largest complement, so that all start from 0).
__global__ void __launch_bounds__(kBlock) k_bucket_sets(const DevSet* __restrict__ sets, uint32_t count,
                                                        const uint64_t* __restrict__ counts,
                                                        uint32_t* __restrict__ bset,
                                                        unsigned long long* __restrict__ cls_max,
                                                        unsigned long long* __restrict__ set_cmin,
                                                        unsigned long long* __restrict__ set_max) {
  const uint32_t si = set_of_block(sets, count, blockIdx.x, 1);
  const DevSet st = sets[si];
  const uint64_t t0 = (blockIdx.x - st.bucket_tile_base) * kTile;
  unsigned long long mx = 0, mn = ~0ull;
  for (int k = 0; k < kTileItems; k++) {
    const uint64_t j = t0 + uint64_t(k) * kBlock + threadIdx.x;
    if (j < st.nb) {
      const uint64_t b = st.bucket_base + j;
      bset[b] = si;
      const unsigned long long c = counts[b];
      mx = max(mx, c);
      mn = min(mn, c);
    }
  }
  for (int o = 16; o; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (mx) {
      atomicMax(cls_max + st.cls, mx);
      atomicMax(set_max + si, mx);
    }
    if (mn != ~0ull) atomicMax(set_cmin + si, ~mn);
  }
}

struct ClassTables {
  const uint64_t* t[kMaxClasses];
  uint64_t mmax[kMaxClasses];  // largest node size of each table
  uint32_t leaf[kMaxClasses];
};

// Sec. 9: grouping by bucket; the order inside a bucket does not matter
// (every search depends on the set only).  Keys are stored as x ^ (x >> 30)
// of their lower half, the form the searches consume.
__global__ void k_scatter(const uint32_t* __restrict__ bucket, const uint64_t* __restrict__ lo, uint64_t n,
                          const uint64_t* __restrict__ bstart, uint32_t* __restrict__ cursor,
                          uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < n; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t b = bucket[i];
    const uint64_t pos = bstart[b] + atomicAdd(cursor + b, 1u);
    out[pos] = pre_key(lo[i]);
  }
}

// Prefix sums over the buckets of all sets of their keys (s_i, bstart), codes
// (first code slot, cbase) and, with RANGE, output ranges (table word 3, upper
// half: the sum of the leaves' ranges), and the first queue entries, in one
// launch: every bucket of two or more keys is appended to the queue of its
// kind (split node, full leaf, partial leaf).  The lanes of a warp that append
// to the same queue take their slots with one atomic: with buckets of a few
// keys there are millions of appends to a handful of counters, and one atomic
// per bucket on the same address serialises them.
constexpr int kGroupItems = 4;
constexpr uint64_t kGroupTile = uint64_t(kBlock) * kGroupItems;

template <bool RANGE>
__global__ void __launch_bounds__(kBlock) k_group_scan(const uint64_t* __restrict__ counts,
                                                       const uint32_t* __restrict__ bset,
                                                       const DevSet* __restrict__ sets, uint64_t nbt, ClassTables ct,
                                                       uint64_t* __restrict__ bstart, uint64_t* __restrict__ cbase,
                                                       uint64_t* __restrict__ rstart, LookState st, SearchArgs a) {
  constexpr int N = RANGE ? 3 : 2;
  __shared__ uint32_t tile_s;
  __shared__ uint64_t before_s[N];
  if (threadIdx.x == 0) tile_s = atomicAdd(st.ticket, 1u);
  __syncthreads();
  const uint32_t tile = tile_s, lane = threadIdx.x & 31;
  const uint64_t base = tile * kGroupTile + threadIdx.x * uint64_t(kGroupItems);
  uint32_t m[kGroupItems], cls[kGroupItems], codes[kGroupItems], range[kGroupItems];
  uint64_t s[N] = {}, run[N], total[N];
#pragma unroll
  for (int k = 0; k < kGroupItems; k++) {
    const uint64_t b = base + k;
    m[k] = cls[k] = codes[k] = range[k] = 0;
    if (b < nbt) {
      m[k] = static_cast<uint32_t>(counts[b]);  // at most 2^32 - 1 keys in all
      cls[k] = sets[bset[b]].cls;
      const uint64_t* t = ct.t[cls[k]] + kTableWords * uint64_t(m[k]);
      codes[k] = static_cast<uint32_t>(t[0] >> 32);
      if (RANGE) range[k] = static_cast<uint32_t>(t[3] >> 32);
    }
    s[0] += m[k];
    s[1] += codes[k];
    if (RANGE) s[N - 1] += range[k];
  }
  block_scan<N, kBlock>(s, run, total);
  if (threadIdx.x < 32) {
    uint64_t before[N];
    look_back<N>(st, tile, total, before, a.error);
    if (threadIdx.x == 0)
      for (int k = 0; k < N; k++) before_s[k] = before[k];
  }
  __syncthreads();
  uint64_t at = run[0] + before_s[0], slot = run[1] + before_s[1], rat = RANGE ? run[N - 1] + before_s[N - 1] : 0;
#pragma unroll
  for (int k = 0; k < kGroupItems; k++) {
    const uint64_t b = base + k;
    if (b < nbt) {
      bstart[b] = at;
      cbase[b] = slot;
      if (RANGE) rstart[b] = rat;
    }
    const bool want = m[k] >= 2;
    const uint32_t active = __ballot_sync(0xFFFFFFFFu, want);
    if (want) {
      const uint32_t c = cls[k], leaf = a.leaf_of[c];
      Node* q;
      uint32_t *cnt, cap;
      if (m[k] > leaf) {
        const int heavy = a.heavy_flag < 2 && heavy_flag(ct.t[c][kTableWords * uint64_t(m[k]) + 1], 0, a.heavy_flag);
        q = a.split_in[heavy], cnt = a.split_in_count[heavy], cap = a.split_cap[heavy];
      } else if (m[k] == leaf)
        q = a.full_q[c], cnt = a.full_n + c, cap = a.full_cap[c];
      else
        q = a.part_q[c], cnt = a.part_n + c, cap = a.part_cap[c];
      const uint32_t peers = __match_any_sync(active, reinterpret_cast<unsigned long long>(cnt));
      const uint32_t leader = __ffs(peers) - 1;
      uint32_t first = 0;
      if (lane == leader) first = atomicAdd(cnt, static_cast<uint32_t>(__popc(peers)));
      first = __shfl_sync(peers, first, leader);
      const uint32_t e = first + __popc(peers & ((1u << lane) - 1));
      if (e < cap)
        q[e] = Node{static_cast<uint32_t>(at), m[k], static_cast<uint32_t>(slot), c << 8};
      else
        atomicCAS(a.error, 0, RECSPLIT_E_INVALID);
    }
    __syncwarp();
    at += m[k];
    slot += codes[k];
    rat += range[k];
  }
  if (threadIdx.x == kBlock - 1 && (tile + 1) * kGroupTile >= nbt) {
    bstart[nbt] = at;
    cbase[nbt] = slot;
    if (RANGE) rstart[nbt] = rat;
  }
}

// ---------------------------------------------------------------- A5
// The kernels over the codes of buckets take a lane per bucket where buckets
// have a few codes and a warp per bucket where they have more: one lane walking
// the 360 codes of a bucket (l = 12, b = 2000) held the lengths of a batched
// build at 0.35 ms and the writing at 0.45 ms.  Lanes are numbered per set from
// a multiple of 32; lane_set finds the set of a warp.
// A warp pays from 64 codes, and from 8 on few buckets, where the time is one
// lane's chain of loads (10 buckets of 18 codes: lengths and writing 9 + 12 -> 4
// + 4 us); on 10^5 such buckets the lanes are the faster (34 us against 81 us,
// for the atomic per code of the warp's writing).  Encode phase with lanes and with
// warps, l = 8: 18 codes a bucket, 1000 buckets 64 and 46 us, 6000 70 and 60, 20000 74 and
// 73, 50000 82 and 95; 36 codes 81 and 47, 88 and 63, 97 and 82, 103 and 110: the line
// could lie at twice to four times as many buckets.
constexpr uint64_t kWarpCodes = 64, kFewWarpCodes = 8, kFewBuckets = 8192;

struct BucketLane {
  uint32_t set;     // ~0: no bucket
  uint64_t bucket;  // global index
  bool whole_warp;
};
__device__ __forceinline__ BucketLane bucket_lane(const DevSet* sets, uint32_t count) {
  const uint64_t t = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x;
  uint32_t lo = 0, hi = count;  // last set with lane_base <= the warp's first lane
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (sets[mid].lane_base <= (t & ~uint64_t(31))) lo = mid; else hi = mid;
  }
  const DevSet& st = sets[lo];
  const bool whole = st.warp_buckets != 0;
  const uint64_t j = (t - st.lane_base) >> (whole ? 5 : 0);
  return BucketLane{t >= st.lane_base && j < st.nb ? lo : ~0u, st.bucket_base + j, whole};
}

// Bits of bucket b: fixed bits of its tree (table) + unary parts (i >> r) + 1.
// After a failed search (error set) the slots of unsearched nodes were never
// written: the lengths are then not computed (the build reports the error).
// Lookups address the bits of a bucket with 32-bit offsets, so a bucket whose
// code reaches 2^32 bits (more than a billion keys in one bucket) fails the
// build with RECSPLIT_E_INVALID.
__global__ void __launch_bounds__(kBlock) k_bucket_bits(const uint64_t* __restrict__ counts,
                                                        const uint64_t* __restrict__ cbase,
                                                        const uint64_t* __restrict__ seeds,
                                                        const uint32_t* __restrict__ sizes,
                                                        const DevSet* __restrict__ sets, uint32_t count,
                                                        ClassTables ct, int* __restrict__ error,
                                                        uint64_t* __restrict__ bits) {
  const bool failed = *reinterpret_cast<const volatile int*>(error) != 0;
  const BucketLane bl = bucket_lane(sets, count);
  if (bl.set == ~0u) return;  // whole warps, or single lanes
  const uint32_t cls = sets[bl.set].cls;
  const uint64_t* table = ct.t[cls];
  const uint64_t mmax = ct.mmax[cls];
  const uint32_t step = bl.whole_warp ? 32 : 1;
  uint64_t len = 0;
  if (!failed)
    for (uint64_t c = cbase[bl.bucket] + (bl.whole_warp ? threadIdx.x & 31 : 0), e = cbase[bl.bucket + 1]; c < e;
         c += step) {
      const uint32_t sz = sizes[c];
      const uint32_t r = sz <= mmax ? static_cast<uint32_t>(table[kTableWords * sz + 1] >> 40) & 31 : 0;
      len += (seeds[c] >> r) + 1;
    }
  if (bl.whole_warp) {
    for (int o = 16; o; o >>= 1) len += __shfl_xor_sync(0xFFFFFFFFu, len, o);
    if (threadIdx.x & 31) return;
  }
  len += static_cast<uint32_t>(table[kTableWords * counts[bl.bucket]]);
  if (!failed && len >= (1ull << 32)) atomicCAS(error, 0, RECSPLIT_E_INVALID);
  bits[bl.bucket] = len;
}

__device__ __forceinline__ uint64_t mulhi32_shift(uint64_t a, uint64_t b) {
  // floor(a * b / 2^32) for a * b < 2^96
  return (__umul64hi(a, b) << 32) | ((a * b) >> 32);
}

__device__ __forceinline__ uint64_t beta_of(uint64_t tree_bits, uint64_t n) {
  // floor(T * 2^32 / n), n < 2^32
  if (n == 0) return 0;
  const uint64_t q = tree_bits / n, r = tree_bits % n;
  return (q << 32) + (r << 32) / n;
}

// Signed 64-bit value as an unsigned one that grows as the value falls, above
// 0: the largest over values that start at 0 is the smallest value.
__host__ __device__ inline unsigned long long falling(long long v) {
  return ~(static_cast<unsigned long long>(v) ^ (1ull << 63));
}

// Per set: the smallest difference of consecutive values o_i - beta s_i (as
// falling()), and its tree bits, codes and output range (differences of the
// global scans at the set's first and one-past-last bucket).
// rstart: prefix sums of the bucket output ranges (of the bucket sizes when
// the leaf range extra is 0), global over all sets.
struct SetResults {
  uint64_t *tree_bits, *codes, *range;
  unsigned long long* delta;  // 0 until the set's buckets are seen
};
__global__ void __launch_bounds__(kBlock) k_ef_prepare(const DevSet* __restrict__ sets, uint32_t count,
                                                       const uint64_t* __restrict__ rstart,
                                                       const uint64_t* __restrict__ off,
                                                       const uint64_t* __restrict__ cbase, SetResults res) {
  const uint32_t si = set_of_block(sets, count, blockIdx.x, 1);
  const DevSet st = sets[si];
  const uint64_t bb = st.bucket_base;
  const uint64_t T = off[bb + st.nb] - off[bb];
  const uint64_t r0 = rstart[bb];
  const uint64_t range = rstart[bb + st.nb] - r0;
  const uint64_t beta = beta_of(T, range);
  const uint64_t t0 = (blockIdx.x - st.bucket_tile_base) * kTile;
  if (t0 == 0 && threadIdx.x == 0) {
    res.tree_bits[si] = T;
    res.codes[si] = cbase[bb + st.nb] - cbase[bb];
    res.range[si] = range;
  }
  long long mn = LLONG_MAX;
  for (int k = 0; k < kTileItems; k++) {
    const uint64_t j = t0 + uint64_t(k) * kBlock + threadIdx.x;
    if (j < st.nb) {
      const long long z0 = (long long)(off[bb + j] - off[bb]) - (long long)mulhi32_shift(rstart[bb + j] - r0, beta);
      const long long z1 =
          (long long)(off[bb + j + 1] - off[bb]) - (long long)mulhi32_shift(rstart[bb + j + 1] - r0, beta);
      mn = min(mn, z1 - z0);
    }
  }
  for (int o = 16; o; o >>= 1) mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
  if ((threadIdx.x & 31) == 0 && mn != LLONG_MAX) atomicMax(res.delta + si, falling(mn));
}

// ---------------------------------------------------------------- A6
__device__ __forceinline__ void or_bits(uint64_t* a, uint64_t pos, uint64_t v, uint32_t width) {
  if (width == 0 || v == 0) return;
  const uint64_t w = pos >> 6;
  const uint32_t o = static_cast<uint32_t>(pos & 63);
  atomicOr(reinterpret_cast<unsigned long long*>(a + w), (unsigned long long)(v << o));
  if (o + width > 64) atomicOr(reinterpret_cast<unsigned long long*>(a + w + 1), (unsigned long long)(v >> (64 - o)));
}

// Bits accumulate per word before an atomic OR, since neighbouring buckets
// share boundary words.
struct BitSink {
  uint64_t* a;
  uint64_t word = ~0ull, acc = 0;
  __device__ void flush() {
    if (word != ~0ull && acc) atomicOr(reinterpret_cast<unsigned long long*>(a + word), (unsigned long long)acc);
    acc = 0;
  }
  __device__ void put(uint64_t pos, uint64_t v, uint32_t width) {
    if (!width) return;
    const uint64_t w = pos >> 6;
    const uint32_t o = static_cast<uint32_t>(pos & 63);
    if (w != word) {
      flush();
      word = w;
    }
    acc |= v << o;
    if (o + width > 64) {
      flush();
      word = w + 1;
      acc = v >> (64 - o);
    }
  }
};

// Per-set output parameters (after the structure layout is known).
struct DevOut {
  uint64_t* blob;
  uint64_t header[kHeaderWords];
  uint64_t* tree;
  uint64_t* lower;
  uint64_t* upper_a;
  uint64_t* upper_b;
  uint64_t* anchors;
  uint16_t* subs;
  uint64_t beta;
  int64_t delta_a, delta_b;
  uint32_t low_a, low_b;
};

// Per bucket: fixed parts of all codes in preorder from o_b, then the unary
// parts from o_b + F(m) (Sec. 6.2).  A warp places 32 codes at a time with
// prefix sums of their fixed and unary lengths.
__global__ void __launch_bounds__(kBlock) k_write_codes(const uint64_t* __restrict__ counts,
                                                        const uint64_t* __restrict__ cbase,
                                                        const uint64_t* __restrict__ seeds,
                                                        const uint32_t* __restrict__ sizes,
                                                        const DevSet* __restrict__ sets, uint32_t count,
                                                        const DevOut* __restrict__ outs, ClassTables ct,
                                                        const uint64_t* __restrict__ off) {
  const BucketLane bl = bucket_lane(sets, count);
  if (bl.set == ~0u) return;  // whole warps, or single lanes
  const uint64_t m = counts[bl.bucket];
  if (m < 2) return;
  const DevSet& st = sets[bl.set];
  const uint64_t* table = ct.t[st.cls];
  const uint64_t mmax = ct.mmax[st.cls];
  uint64_t* tree = outs[bl.set].tree;
  const uint64_t base = off[bl.bucket] - off[st.bucket_base];
  uint64_t fpos = base;
  uint64_t upos = base + static_cast<uint32_t>(table[kTableWords * m]);
  const uint64_t first = cbase[bl.bucket], e = cbase[bl.bucket + 1];
  if (!bl.whole_warp) {
    BitSink fixed{tree}, unary{tree};
    for (uint64_t c = first; c < e; c++) {
      const uint32_t sz = sizes[c];
      const uint32_t r = sz <= mmax ? static_cast<uint32_t>(table[kTableWords * sz + 1] >> 40) & 31 : 0;
      const uint64_t s = seeds[c];
      fixed.put(fpos, r ? (s & ((1ull << r) - 1)) : 0, r);
      fpos += r;
      upos += s >> r;
      unary.put(upos, 1, 1);
      upos++;
    }
    fixed.flush();
    unary.flush();
    return;
  }
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t c0 = first; c0 < e; c0 += 32) {
    const uint64_t c = c0 + lane;
    uint32_t r = 0;
    uint64_t s = 0, u = 0;  // unary length
    if (c < e) {
      const uint32_t sz = sizes[c];
      r = sz <= mmax ? static_cast<uint32_t>(table[kTableWords * sz + 1] >> 40) & 31 : 0;
      s = seeds[c];
      u = (s >> r) + 1;
    }
    uint32_t fr = r;
    uint64_t ur = u;
    for (uint32_t d = 1; d < 32; d <<= 1) {
      const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, fr, d);
      const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, ur, d);
      if (lane >= d) {
        fr += x;
        ur += y;
      }
    }
    if (c < e) {
      or_bits(tree, fpos + fr - r, r ? (s & ((1ull << r) - 1)) : 0, r);
      or_bits(tree, upos + ur - 1, 1, 1);
    }
    fpos += __shfl_sync(0xFFFFFFFFu, fr, 31);
    upos += __shfl_sync(0xFFFFFFFFu, ur, 31);
  }
}

// ---------------------------------------------------------------- A7
__device__ __forceinline__ void ef_values(const DevSet& st, const DevOut& p, const uint64_t* rstart,
                                          const uint64_t* off, uint64_t i, uint64_t& xa, uint64_t& xb) {
  const uint64_t s = rstart[st.bucket_base + i] - rstart[st.bucket_base];
  const int64_t z = (int64_t)(off[st.bucket_base + i] - off[st.bucket_base]) - (int64_t)mulhi32_shift(s, p.beta);
  xa = s - static_cast<uint64_t>((int64_t)i * p.delta_a);
  xb = static_cast<uint64_t>(z - (int64_t)i * p.delta_b);
}

// Elements 0 .. nb of every set: interleaved lower bits, upper bits, and the
// u64 / u16 inventories of both lists; and the header (every set has an
// element, so a first block).
__global__ void __launch_bounds__(kBlock) k_ef_write(const DevSet* __restrict__ sets, uint32_t count,
                                                     const DevOut* __restrict__ outs,
                                                     const uint64_t* __restrict__ rstart,
                                                     const uint64_t* __restrict__ off) {
  const uint32_t si = set_of_block(sets, count, blockIdx.x, 2);
  const DevSet st = sets[si];
  const DevOut& p = outs[si];
  const uint64_t t0 = (blockIdx.x - st.elem_tile_base) * kTile;
  if (t0 == 0 && threadIdx.x < kHeaderWords) p.blob[threadIdx.x] = p.header[threadIdx.x];
  for (int k = 0; k < kTileItems; k++) {
    const uint64_t i = t0 + uint64_t(k) * kBlock + threadIdx.x;
    if (i > st.nb) break;
    uint64_t xa, xb;
    ef_values(st, p, rstart, off, i, xa, xb);
    const uint64_t rec = i * (p.low_a + p.low_b);
    or_bits(p.lower, rec, p.low_a ? (xa & ((1ull << p.low_a) - 1)) : 0, p.low_a);
    or_bits(p.lower, rec + p.low_a, p.low_b ? (xb & ((1ull << p.low_b) - 1)) : 0, p.low_b);
    const uint64_t pa = (xa >> p.low_a) + i, pb = (xb >> p.low_b) + i;
    or_bits(p.upper_a, pa, 1, 1);
    or_bits(p.upper_b, pb, 1, 1);
    if ((i & ((1u << kInvHi) - 1)) == 0) {
      p.anchors[2 * (i >> kInvHi)] = pa;
      p.anchors[2 * (i >> kInvHi) + 1] = pb;
    }
    if ((i & ((1u << kInvLo) - 1)) == 0) {
      const uint64_t a0 = (i >> kInvHi) << kInvHi;
      uint64_t ya, yb;
      ef_values(st, p, rstart, off, a0, ya, yb);
      const uint64_t da = pa - ((ya >> p.low_a) + a0), db = pb - ((yb >> p.low_b) + a0);
      p.subs[2 * (i >> kInvLo)] = static_cast<uint16_t>(da < 0xFFFF ? da : 0xFFFF);
      p.subs[2 * (i >> kInvLo) + 1] = static_cast<uint16_t>(db < 0xFFFF ? db : 0xFFFF);
    }
  }
}

// ---------------------------------------------------------------- tracing
// Algorithmic work of the searches: per code slot, (index + 1) trials of
// `size` evaluations each, summed separately for splits and leaves.
__global__ void k_work(const uint64_t* __restrict__ seeds, const uint32_t* __restrict__ sizes,
                       const uint64_t* __restrict__ ncodes_p, const uint32_t* __restrict__ code_leaf,
                       unsigned long long* __restrict__ sums) {
  const uint64_t ncodes = *ncodes_p;
  unsigned long long v[6] = {0, 0, 0, 0, 0, 0};
  for (uint64_t c = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; c < ncodes; c += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t t = seeds[c] + 1, m = sizes[c];
    const int k = m > code_leaf[c] ? 0 : 3;
    v[k] += 1;
    v[k + 1] += t;
    v[k + 2] += t * m;
  }
#pragma unroll
  for (int k = 0; k < 6; k++) {
    for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
    if ((threadIdx.x & 31) == 0 && v[k]) atomicAdd(sums + k, v[k]);
  }
}

// Leaf size of each code slot (for the split/leaf split of the work counts).
__global__ void k_code_leaf(const uint64_t* __restrict__ cbase, const uint32_t* __restrict__ bset,
                            const DevSet* __restrict__ sets, uint64_t nbt, uint32_t* __restrict__ code_leaf) {
  for (uint64_t b = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; b < nbt; b += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t leaf = sets[bset[b]].leaf;
    for (uint64_t c = cbase[b], e = cbase[b + 1]; c < e; c++) code_leaf[c] = leaf;
  }
}

// Phase boundaries of a build: CUDA events on the build stream when
// profiling is on, and always an NVTX range per phase (named
// recsplit.signature, .group, .split, .leaves, .encode) around the launches
// of that phase, so that a profiler can select one phase's kernels.
struct PhaseTimer {
  static constexpr const char* kNames[5] = {"recsplit.signature", "recsplit.group", "recsplit.split",
                                            "recsplit.leaves", "recsplit.encode"};
  bool on;
  cudaStream_t s;
  cudaEvent_t ev[6] = {};
  int k = 0;
  int ranges = 0;  // marks seen; a range is open while 1 <= ranges <= 5
  PhaseTimer(bool enabled, cudaStream_t stream) : on(enabled), s(stream) {
    if (on)
      for (auto& e : ev) cudaEventCreate(&e);
  }
  ~PhaseTimer() {
    if (ranges >= 1 && ranges <= 5) nvtxRangePop();
    if (on)
      for (auto& e : ev) cudaEventDestroy(e);
  }
  void mark() {
    if (ranges >= 1 && ranges <= 5) nvtxRangePop();
    if (ranges < 5) nvtxRangePushA(kNames[ranges]);
    ranges++;
    if (on && k < 6) cudaEventRecord(ev[k++], s);
  }
  double ms(int a, int b) const {
    float t = 0.f;
    if (on && b < k) cudaEventElapsedTime(&t, ev[a], ev[b]);
    return t;
  }
};

// ---------------------------------------------------------------- host
// Stream-ordered scratch of a build.  plan() lists the arrays of one
// allocation (256-byte aligned each) and alloc() makes it: the small per-bucket
// and per-set arrays share allocations, since thirty of them, and as many
// frees, took about a tenth of the time of a build of 10^3 keys.
struct Scratch {
  cudaStream_t s;
  std::vector<void*> ptrs;
  std::vector<std::pair<void**, size_t>> planned;
  size_t bytes = 0;
  ~Scratch() {
    for (void* p : ptrs) cudaFreeAsync(p, s);
  }
  template <typename T>
  void plan(T** p, uint64_t count) {
    planned.emplace_back(reinterpret_cast<void**>(p), bytes);
    bytes += (std::max<uint64_t>(count, 1) * sizeof(T) + 255) & ~size_t(255);
  }
  // `zero` set: the whole allocation starts as zeros
  int alloc(bool zero = false) {
    void* q = nullptr;
    const size_t n = bytes;
    std::vector<std::pair<void**, size_t>> list;
    list.swap(planned);
    bytes = 0;
    int rc = pool_alloc(&q, n, s);
    if (rc) return rc;
    ptrs.push_back(q);
    for (auto& e : list) *e.first = static_cast<char*>(q) + e.second;
    if (zero) RS_CUDA(cudaMemsetAsync(q, 0, n, s));
    return RECSPLIT_OK;
  }
  template <typename T>
  int alloc(T** p, uint64_t count) {
    plan(p, count);
    return alloc();
  }
};

// Results a build reads back from the device: one copy, into page-locked
// memory of the host thread where they fit (a copy to pageable memory waits
// for the stream by itself and is staged).
struct Readback {
  static constexpr size_t kBytes = 64 << 10;
  struct Pinned {
    void* p = nullptr;
    bool tried = false;
    ~Pinned() {
      if (p) cudaFreeHost(p);
    }
  };
  std::vector<uint64_t> pageable;
  uint64_t* words = nullptr;
  bool pinned = false;
  explicit Readback(size_t n) {
    static thread_local Pinned mine;
    if (!mine.tried) {
      mine.tried = true;
      if (cudaHostAlloc(&mine.p, kBytes, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        mine.p = nullptr;
      }
    }
    pinned = mine.p && n * sizeof(uint64_t) <= kBytes;
    if (!pinned) pageable.resize(n);
    words = pinned ? static_cast<uint64_t*>(mine.p) : pageable.data();
  }
};

int floor_log2_u64(uint64_t x) { return x ? 63 - __builtin_clzll(x) : 0; }

int ef_width(uint64_t u, uint64_t count) {
  const uint64_t q = u / count;
  return q ? floor_log2_u64(q) : 0;
}

uint64_t tiles(uint64_t items) { return (items + kTile - 1) / kTile; }

// Parameter class of a set.
uint32_t class_key(const SetInput& si) { return si.leaf | (si.leaf_extra << 8); }

// Adds the profile of a pass to the call's.
void add_profile(recsplit_profile_t* sum, const recsplit_profile_t& p) {
  sum->ms_signature += p.ms_signature;
  sum->ms_group += p.ms_group;
  sum->ms_split += p.ms_split;
  sum->ms_leaf += p.ms_leaf;
  sum->ms_encode += p.ms_encode;
  sum->ms_total += p.ms_total;
  sum->split_nodes += p.split_nodes;
  sum->split_trials += p.split_trials;
  sum->split_evals += p.split_evals;
  sum->leaf_nodes += p.leaf_nodes;
  sum->leaf_trials += p.leaf_trials;
  sum->leaf_evals += p.leaf_evals;
  sum->launches += p.launches;
  sum->split_levels += p.split_levels;
  sum->leaf_evals_executed += p.leaf_evals_executed;
  sum->split_evals_executed += p.split_evals_executed;
}

}  // namespace

// One pass over sets of at most kMaxClasses classes; t_call: start of the call
// (time limit).
static int build_pass(const SetInput* in, uint32_t count, const BuildOptions& opt, cudaStream_t s, double t_call,
                      Handle** out) {
  int dev = 0, sm_count = 0;
  RS_CUDA(cudaGetDevice(&dev));
  RS_CUDA(cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev));

  // ---- host plan: classes (distinct leaf sizes and leaf range extras), bases, tilings
  std::map<uint32_t, uint32_t> cls_of_leaf;
  std::vector<uint32_t> class_leaf, class_extra;
  bool any_extra = false;
  std::vector<DevSet> hs(count);
  uint64_t K = 0, NB = 0, key_tiles = 0, bucket_tiles = 0, elem_tiles = 0;
  for (uint32_t i = 0; i < count; i++) {
    const SetInput& si = in[i];
    any_extra |= si.leaf_extra != 0;
    const uint32_t key = class_key(si);
    auto it = cls_of_leaf.find(key);
    if (it == cls_of_leaf.end()) {
      it = cls_of_leaf.emplace(key, static_cast<uint32_t>(class_leaf.size())).first;
      class_leaf.push_back(si.leaf);
      class_extra.push_back(si.leaf_extra);
    }
    DevSet& d = hs[i];
    d.u64 = si.keys.u64;
    d.bytes = si.keys.bytes;
    d.offsets = si.keys.offsets;
    d.n = si.keys.n;
    d.key_base = K;
    d.nb = (d.n + si.bucket_size - 1) / si.bucket_size;
    d.bucket_base = NB;
    d.cls = it->second;
    d.leaf = si.leaf;
    d.key_tile_base = key_tiles;
    d.bucket_tile_base = bucket_tiles;
    d.elem_tile_base = elem_tiles;
    K += d.n;
    NB += d.nb;
    key_tiles += tiles(d.n);
    bucket_tiles += tiles(d.nb);
    elem_tiles += tiles(d.nb + 1);
  }
  const uint32_t nclass = static_cast<uint32_t>(class_leaf.size());

  // classes by key count (queue capacities): a split node has more keys than
  // its leaf size, and each split node or bucket yields at most one partial leaf
  std::vector<uint64_t> keys_c(nclass, 0), nb_c(nclass, 0), full_cap(nclass), part_cap(nclass);
  for (const DevSet& d : hs) {
    keys_c[d.cls] += d.n;
    nb_c[d.cls] += d.nb;
  }
  uint64_t split_cap = 1, qtotal = 0;
  for (uint32_t c = 0; c < nclass; c++) {
    split_cap += keys_c[c] / (class_leaf[c] + 1);
    full_cap[c] = keys_c[c] / class_leaf[c] + 1;
    part_cap[c] = nb_c[c] + keys_c[c] / (class_leaf[c] + 1) + 1;
    qtotal += full_cap[c] + part_cap[c];
  }

  Scratch sc{s};
  PhaseTimer timer(profiling_enabled(), s);
  const uint64_t launch0 = launch_mark();
  uint32_t split_levels = 0;
  timer.mark();
  int rc;
  const bool count_work = timer.on && work_counting_enabled();
  // what starts as zeros, in one allocation and one memset
  uint64_t* counts;
  uint32_t *cursor, *sizes;
  uint64_t* back1;  // read back after the histogram: class maxima, bad offsets, set minima (complements), set maxima
  uint64_t* back2;  // and after the lengths: tree bits, codes, ranges, smallest deltas, error
  const uint64_t n_back1 = kMaxClasses + 1 + 2 * uint64_t(count), n_back2 = 4 * uint64_t(count) + 1;
  // one counter per use, so that none is zeroed between launches: nodes of
  // every split level, work counters of the split and leaf launches, leaves
  constexpr uint32_t kLevels = kMaxDepth + 3;
  uint32_t* counters;
  unsigned long long* exec = nullptr;  // work counting: evaluations executed
  sc.plan(&counts, NB + 1);
  sc.plan(&cursor, NB + 1);
  sc.plan(&sizes, K + 1);
  sc.plan(&back1, n_back1);
  sc.plan(&back2, n_back2);
  sc.plan(&counters, 4 * kLevels + 4 * kMaxClasses + 2);
  // scans: group_scan's tiles, then those of the lengths
  const uint64_t group_tiles = (NB + kGroupTile - 1) / kGroupTile, bit_tiles = scan_tiles(NB);
  uint32_t* look_flags;
  sc.plan(&look_flags, group_tiles + bit_tiles);
  if (count_work) sc.plan(&exec, 2);
  if ((rc = sc.alloc(/*zero=*/true))) return rc;
  unsigned long long* cls_max = reinterpret_cast<unsigned long long*>(back1);
  int* bad_offsets = reinterpret_cast<int*>(back1 + kMaxClasses);
  unsigned long long* set_cmin = cls_max + kMaxClasses + 1;
  unsigned long long* set_max = set_cmin + count;
  SetResults results{back2, back2 + count, back2 + 2 * uint64_t(count),
                     reinterpret_cast<unsigned long long*>(back2 + 3 * uint64_t(count))};
  int* d_error = reinterpret_cast<int*>(back2 + 4 * uint64_t(count));
  uint32_t* const level_n = counters;                     // split nodes per level, light and heavy
  uint32_t* const level_work = counters + 2 * kLevels;    // and the work counters of its launches
  uint32_t* const leaf_work = level_work + 2 * kLevels;   // two leaf launches per class
  uint32_t* const full_n = leaf_work + 2 * kMaxClasses;
  uint32_t* const part_n = full_n + kMaxClasses;
  uint32_t* const tickets = part_n + kMaxClasses;

  DevSet* d_sets;
  DevOut* d_outs;
  uint32_t *bucket, *bset;
  uint64_t *lo, *bstart, *cbase, *bits, *off, *look;
  // prefix sums of the bucket output ranges: s_i itself unless a set has a
  // leaf range extra
  uint64_t* rstart = nullptr;
  sc.plan(&d_sets, count);
  sc.plan(&d_outs, count);
  if ((rc = sc.alloc())) return rc;
  sc.plan(&bstart, NB + 1);
  sc.plan(&cbase, NB + 1);
  sc.plan(&bset, NB + 1);
  sc.plan(&bits, NB + 1);
  sc.plan(&off, NB + 1);
  sc.plan(&look, 6 * std::max(group_tiles, bit_tiles));
  if (any_extra) sc.plan(&rstart, NB + 1);
  if ((rc = sc.alloc()) || (rc = sc.alloc(&bucket, K)) || (rc = sc.alloc(&lo, K))) return rc;
  if (!any_extra) rstart = bstart;
  RS_CUDA(cudaMemcpyAsync(d_sets, hs.data(), count * sizeof(DevSet), cudaMemcpyHostToDevice, s));

  // A1 + A2: signatures, bucket ids, histogram; bucket -> set; extremes
  if (key_tiles) {
    k_signature<<<static_cast<unsigned>(key_tiles), kBlock, 0, s>>>(
        d_sets, count, bucket, lo, reinterpret_cast<unsigned long long*>(counts), bad_offsets);
    count_launch();
  }
  if (bucket_tiles) {
    k_bucket_sets<<<static_cast<unsigned>(bucket_tiles), kBlock, 0, s>>>(d_sets, count, counts, bset, cls_max,
                                                                         set_cmin, set_max);
    count_launch();
  }
  RS_CUDA(cudaGetLastError());
  timer.mark();
  std::vector<uint64_t> h_cls_max(kMaxClasses), h_set_min(count), h_set_max(count);
  {
    Readback back(n_back1);
    RS_CUDA(cudaMemcpyAsync(back.words, back1, n_back1 * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    RS_CUDA(cudaStreamSynchronize(s));  // sync 1: largest bucket per class
    if (static_cast<int>(back.words[kMaxClasses])) return fail(RECSPLIT_E_INVALID, "byte-string offsets must not decrease");
    std::copy_n(back.words, kMaxClasses, h_cls_max.begin());
    for (uint32_t i = 0; i < count; i++) h_set_min[i] = ~back.words[kMaxClasses + 1 + i];
    std::copy_n(back.words + kMaxClasses + 1 + count, count, h_set_max.begin());
  }

  // tables per class, in one buffer
  std::vector<Tables> T(nclass);
  std::vector<uint64_t> tbase(nclass + 1, 0);
  std::string err;
  for (uint32_t c = 0; c < nclass; c++) {
    if ((rc = build_tables(class_leaf[c], class_extra[c], h_cls_max[c], &T[c], &err))) return fail(rc, err);
    tbase[c + 1] = tbase[c] + T[c].device_words.size();
  }
  auto table_mem = std::make_shared<DeviceMem>();
  if ((rc = pool_alloc(&table_mem->p, tbase[nclass] * sizeof(uint64_t), s))) return rc;
  uint64_t* d_tables = static_cast<uint64_t*>(table_mem->p);
  {
    std::vector<uint64_t> all(tbase[nclass]);
    for (uint32_t c = 0; c < nclass; c++)
      std::copy(T[c].device_words.begin(), T[c].device_words.end(), all.begin() + tbase[c]);
    RS_CUDA(cudaMemcpyAsync(d_tables, all.data(), all.size() * sizeof(uint64_t), cudaMemcpyHostToDevice, s));
  }
  ClassTables ct{};
  for (uint32_t c = 0; c < nclass; c++) {
    ct.t[c] = d_tables + tbase[c];
    ct.mmax[c] = T[c].mmax;
    ct.leaf[c] = class_leaf[c];
  }

  // lanes of the kernels over codes: by the codes of a mean bucket
  uint64_t lanes = 0;
  for (uint32_t i = 0; i < count; i++) {
    DevSet& d = hs[i];
    const uint64_t mean = d.nb ? std::min(T[d.cls].mmax, d.n / d.nb) : 0;
    d.warp_buckets = T[d.cls].codes[mean] >= (NB <= kFewBuckets ? kFewWarpCodes : kWarpCodes);
    d.lane_base = lanes;
    lanes += d.warp_buckets ? d.nb * 32 : (d.nb + 31) & ~uint64_t(31);
  }
  RS_CUDA(cudaMemcpyAsync(d_sets, hs.data(), count * sizeof(DevSet), cudaMemcpyHostToDevice, s));

  // Heavy nodes are searched shared: that costs a few microseconds of CTA-wide
  // steps per node and removes the tail of a level, a few long geometric
  // searches on an idle device, so it pays where a node's expected trials x keys
  // reach 2^21 evaluations, or 2^16 in a build of few such nodes: 8 per warp of
  // the device, counting the keys of a class over its smallest such node.
  // Split phase without and with the second clause: l = 12, b = 100: 10^5 keys
  // 0.84 -> 0.31 ms, 10^6 keys 2.29 -> 1.69 ms (5 * 10^6 keys, above the line: 7.1
  // against 8.2 ms); l = 13, b = 100, 3 * 10^5 keys 12.6 -> 4.5 ms; l = 16, b = 100, 3 *
  // 10^4 keys 26 -> 5.4 ms; l = 12, b = 2000, 3 * 10^5 keys 4.7 -> 2.1 ms.  Light nodes of
  // the same level have a queue of their own (48 sets with l = 5, 8, 12: all
  // nodes of four such levels shared took 9.2 ms, the heavy ones alone 7.2).
  std::vector<uint64_t> level_max(nclass);
  uint32_t max_leaf = 0;
  double heavy_keys = 0;  // keys over the smallest node of 2^16
  bool any_heavy = false;
  for (uint32_t c = 0; c < nclass; c++) {
    level_max[c] = h_cls_max[c];
    max_leaf = std::max(max_leaf, class_leaf[c]);
    if (h_cls_max[c] <= class_leaf[c] || T[c].heaviest[h_cls_max[c]] < double(kHeavyEvals[0])) continue;
    any_heavy = true;
    const auto& hv = T[c].heaviest;
    heavy_keys += double(keys_c[c]) / double(std::lower_bound(hv.begin(), hv.end(), double(kHeavyEvals[0])) - hv.begin());
  }
  const uint32_t heavy_flag_index = heavy_keys <= 8.0 * 32 * sm_count ? 0 : 1;
  const uint64_t heavy_min = kHeavyEvals[heavy_flag_index];
  // the levels that may hold heavy nodes: sizes that occur, from the bucket
  // sizes down
  std::vector<char> level_heavy;
  if (any_heavy) {
    std::vector<std::vector<uint32_t>> sizes_at(nclass);
    for (uint32_t c = 0; c < nclass; c++) {
      if (T[c].heaviest[h_cls_max[c]] < double(heavy_min)) continue;
      uint64_t least = h_cls_max[c];
      for (uint32_t i = 0; i < count; i++)
        if (hs[i].cls == c && hs[i].nb) least = std::min(least, h_set_min[i]);
      for (uint64_t m = std::max<uint64_t>(least, class_leaf[c] + 1); m <= h_cls_max[c]; m++)
        sizes_at[c].push_back(static_cast<uint32_t>(m));
    }
    std::vector<char> seen;
    for (bool some = true; some && level_heavy.size() <= kMaxDepth + 1;) {
      bool heavy = false;
      some = false;
      for (uint32_t c = 0; c < nclass; c++) {
        if (sizes_at[c].empty()) continue;
        const Strategy st = make_strategy(class_leaf[c]);
        seen.assign(h_cls_max[c] + 1, 0);
        std::vector<uint32_t> next;
        for (uint32_t m : sizes_at[c]) {
          const uint64_t e = T[c].expected_trials[m];
          heavy |= is_heavy(e, m, heavy_min);
          const Shape sh = shape_of(st, m);
          for (uint64_t k : {sh.unit, sh.last})
            if (k > class_leaf[c] && !seen[k]) {
              seen[k] = 1;
              next.push_back(static_cast<uint32_t>(k));
            }
        }
        sizes_at[c].swap(next);
        some |= !sizes_at[c].empty();
      }
      level_heavy.push_back(heavy);
    }
  }
  // heavy nodes of a level hold disjoint keys, each at least as many as the
  // smallest heavy node of its class (with a queue as long as the light nodes', and
  // its search state, a build of 2 * 10^7 keys at l = 12, b = 100 took 48.7 bytes per
  // key, 45.3 so)
  uint64_t heavy_cap = 0;
  for (uint32_t c = 0; c < nclass; c++)
    for (uint64_t m = class_leaf[c] + 1; m <= h_cls_max[c]; m++)
      if (is_heavy(T[c].expected_trials[m], m, heavy_min)) {
        heavy_cap += keys_c[c] / m;
        break;
      }
  qtotal += 2 * (split_cap + heavy_cap);

  // grouping; queues: two split levels (ping-pong) shared by all classes, full
  // and partial leaves per class
  uint64_t* keys[2];
  Node* qmem;
  uint64_t* seeds;
  if ((rc = sc.alloc(&keys[0], K)) || (rc = sc.alloc(&keys[1], K)) || (rc = sc.alloc(&qmem, qtotal)) ||
      (rc = sc.alloc(&seeds, K + 1)))
    return rc;
  SearchArgs a{};
  a.keys[0] = keys[0];
  a.keys[1] = keys[1];
  a.seeds = seeds;
  a.sizes = sizes;
  Node* q_split[2][2] = {{qmem, qmem + split_cap}, {qmem + 2 * split_cap, qmem + 2 * split_cap + heavy_cap}};
  {
    Node* q = qmem + 2 * (split_cap + heavy_cap);
    for (uint32_t c = 0; c < nclass; c++) {
      a.table[c] = ct.t[c];
      a.leaf_of[c] = class_leaf[c];
      a.extra_of[c] = class_extra[c];
      a.full_q[c] = q;
      a.full_cap[c] = static_cast<uint32_t>(full_cap[c]);
      q += full_cap[c];
      a.part_q[c] = q;
      a.part_cap[c] = static_cast<uint32_t>(part_cap[c]);
      q += part_cap[c];
    }
  }
  a.split_cap[0] = static_cast<uint32_t>(split_cap);
  a.split_cap[1] = static_cast<uint32_t>(heavy_cap);
  a.heavy_flag = any_heavy ? heavy_flag_index : 2;
  a.full_n = full_n;
  a.part_n = part_n;
  a.error = d_error;
  a.exec_count = exec;
  for (int h = 0; h < 2; h++) {
    a.split_in[h] = q_split[h][0];
    a.split_in_count[h] = level_n + h;
  }
  // prefix sums s_i, code-slot bases (global over all sets), first queue entries
  if (NB) {
    const LookState st{look_flags, look, look + 3 * std::max(group_tiles, bit_tiles), tickets};
    (any_extra ? k_group_scan<true> : k_group_scan<false>)<<<static_cast<unsigned>(group_tiles), kBlock, 0, s>>>(
        counts, bset, d_sets, NB, ct, bstart, cbase, rstart, st, a);
    count_launch();
  } else {
    RS_CUDA(cudaMemsetAsync(bstart, 0, sizeof(uint64_t), s));
    RS_CUDA(cudaMemsetAsync(cbase, 0, sizeof(uint64_t), s));
    RS_CUDA(cudaMemsetAsync(rstart, 0, sizeof(uint64_t), s));
  }
  if (K) {
    k_scatter<<<std::min<unsigned>(grid_for(K), sm_count * 16), kBlock, 0, s>>>(bucket, lo, K, bstart, cursor,
                                                                                 keys[0]);
    count_launch();
  }
  RS_CUDA(cudaGetLastError());
  timer.mark();

  SharedNodes shared{};
  uint64_t share_cap = heavy_cap;
  std::vector<char> share_leaves(nclass);
  for (uint32_t c = 0; c < nclass; c++) {
    share_leaves[c] = leaves_shared(class_leaf[c], class_extra[c]);
    if (share_leaves[c]) share_cap = std::max(share_cap, full_cap[c]);
  }
  if (share_cap) {
    // (flag and owned are zeroed once: every launch has its own epoch)
    sc.plan(&shared.flag, share_cap);
    sc.plan(&shared.owned, kSharedCtas);
    if ((rc = sc.alloc(/*zero=*/true))) return rc;
    sc.plan(&shared.best, share_cap);
    sc.plan(&shared.next, share_cap);
    sc.plan(&shared.refs, share_cap);
    sc.plan(&shared.cap, share_cap);
    if ((rc = sc.alloc())) return rc;
  }

  // A3 (split levels), A4 (leaves), A5 (lengths): optionally one CUDA graph
  // The graph is captured on a stream of its own (the caller's stream may be
  // the legacy default stream, which cannot be captured) and launched on s.
  cudaGraph_t graph = nullptr;
  cudaStream_t ws = s;
  struct StreamGuard {
    cudaStream_t st = nullptr;
    ~StreamGuard() {
      if (st) cudaStreamDestroy(st);
    }
  } capture_stream;
  if (opt.use_graph) {
    RS_CUDA(cudaStreamCreateWithFlags(&capture_stream.st, cudaStreamNonBlocking));
    ws = capture_stream.st;
    RS_CUDA(cudaStreamBeginCapture(ws, cudaStreamCaptureModeThreadLocal));
  }
  auto search_phase = [&]() -> int {
    int level = 0;
    for (;;) {
      uint64_t mx = 0, trials = 0;
      bool tables = false;  // nodes of five leaves or more, split in equal parts (leaf sizes from 11)
      for (uint32_t c = 0; c < nclass; c++)
        if (level_max[c] > class_leaf[c]) {
          mx = std::max(mx, level_max[c]);
          trials = std::max(trials, T[c].expected_trials[level_max[c]]);
          tables |= class_leaf[c] >= 11 && level_max[c] >= 5 * class_leaf[c];
        }
      if (mx == 0) break;
      if (level > kMaxDepth) return fail(RECSPLIT_E_INVALID, "splitting tree deeper than 63 levels");
      const int cur = level & 1;
      for (int h = 0; h < 2; h++) {
        a.split_in[h] = q_split[h][cur];
        a.split_in_count[h] = level_n + 2 * level + h;
        a.split_out[h] = q_split[h][cur ^ 1];
        a.split_out_count[h] = level_n + 2 * (level + 1) + h;
      }
      a.work_counter = level_work + 2 * level;
      int r = launch_split_level(a, mx, trials, max_leaf, tables, sm_count, ws);
      if (!r && size_t(level) < level_heavy.size() && level_heavy[level]) {
        a.work_counter++;
        shared.epoch++;
        r = launch_split_level(a, mx, trials, max_leaf, tables, sm_count, ws, &shared);
      }
      if (r) return r;
      for (uint32_t c = 0; c < nclass; c++)
        level_max[c] = level_max[c] > class_leaf[c] ? T[c].next_max[level_max[c]] : 0;
      level++;
      split_levels++;
    }
    if (!opt.use_graph) timer.mark();
    for (uint32_t c = 0; c < nclass; c++) {
      a.cls = c;
      a.work_counter = leaf_work + 2 * c;
      if (share_leaves[c]) shared.epoch++;
      int r = launch_leaves(a, class_leaf[c], class_extra[c], h_cls_max[c], sm_count, ws,
                            share_leaves[c] ? &shared : nullptr);
      if (r) return r;
    }
    if (!opt.use_graph) timer.mark();
    if (NB) {
      k_bucket_bits<<<grid_for(lanes), kBlock, 0, ws>>>(counts, cbase, seeds, sizes, d_sets, count, ct, d_error, bits);
      count_launch();
    }
    const LookState st{look_flags + group_tiles, look, look + 3 * std::max(group_tiles, bit_tiles), tickets + 1};
    int r = exclusive_scan_u64(bits, off, NB, st, d_error, ws);
    if (r) return r;
    if (bucket_tiles) {
      k_ef_prepare<<<static_cast<unsigned>(bucket_tiles), kBlock, 0, ws>>>(d_sets, count, rstart, off, cbase, results);
      count_launch();
    }
    RS_CUDA(cudaGetLastError());
    return RECSPLIT_OK;
  };
  rc = search_phase();
  if (opt.use_graph) {
    cudaError_t e = cudaStreamEndCapture(ws, &graph);
    if (rc) {
      if (graph) cudaGraphDestroy(graph);
      return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e, "graph capture");
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(e, "graph instantiation");
    e = cudaGraphLaunch(exec, s);
    cudaGraphExecDestroy(exec);
    if (e != cudaSuccess) return cuda_fail(e, "graph launch");
    timer.mark();
    timer.mark();
  } else if (rc) {
    return rc;
  }

  // sync 2: per-set tree size and minimum delta of the offsets list
  std::vector<long long> h_db(count, 0);
  std::vector<uint64_t> h_T(count), h_codes(count), h_R(count);
  int herr = 0;
  {
    // the deadline wait comes before a copy into pageable memory, which would
    // itself wait for the whole search
    Readback back(n_back2);
    if (!back.pinned && (rc = wait_stream(s, d_error, timeout_ms(), t_call))) return rc;
    RS_CUDA(cudaMemcpyAsync(back.words, back2, n_back2 * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    if (back.pinned)
      rc = wait_stream(s, d_error, timeout_ms(), t_call);
    else
      RS_CUDA(cudaStreamSynchronize(s));
    if (rc) return rc;
    std::copy_n(back.words, count, h_T.begin());
    std::copy_n(back.words + count, count, h_codes.begin());
    std::copy_n(back.words + 2 * uint64_t(count), count, h_R.begin());
    for (uint32_t i = 0; i < count; i++)
      if (const uint64_t d = back.words[3 * uint64_t(count) + i]) h_db[i] = static_cast<long long>(~d ^ (1ull << 63));
    herr = static_cast<int>(back.words[4 * uint64_t(count)]);
  }
  if (herr == RECSPLIT_E_DUPLICATE) return fail(herr, "two keys share their lower signature half (duplicate keys)");
  if (herr == RECSPLIT_E_SEARCH_LIMIT) return fail(herr, "seed search exceeded its limit");
  if (herr) return fail(herr, "a queue capacity, bucket code length or prefix sum check failed");

  // headers and layouts; one arena for all structures (256-byte aligned each)
  std::vector<uint64_t> headers(uint64_t(count) * kHeaderWords, 0), blob_off(count + 1, 0);
  std::vector<DevOut> houts(count);
  std::vector<Layout> layouts(count);
  for (uint32_t i = 0; i < count; i++) {
    const DevSet& d = hs[i];
    uint64_t* H = headers.data() + uint64_t(i) * kHeaderWords;
    const uint64_t n = d.n, nb = d.nb;
    // the first list holds the prefix sums of the bucket output ranges (the
    // bucket sizes unless the set has a leaf range extra); nr is their total
    const uint64_t nr = h_R[i];
    const uint64_t T_bits = h_T[i];
    const uint64_t beta = nr ? ((T_bits / nr) << 32) + (((T_bits % nr) << 32) / nr) : 0;
    const int64_t delta_a = nb ? static_cast<int64_t>(T[d.cls].range[h_set_min[i]]) : 0;
    const int64_t delta_b = nb ? static_cast<int64_t>(h_db[i]) : 0;
    const uint64_t xa_last = nr - static_cast<uint64_t>(static_cast<int64_t>(nb) * delta_a);
    const uint64_t z_last = T_bits - static_cast<uint64_t>((static_cast<unsigned __int128>(nr) * beta) >> 32);
    const uint64_t xb_last = static_cast<uint64_t>(static_cast<int64_t>(z_last) - static_cast<int64_t>(nb) * delta_b);
    const int la = ef_width(xa_last, nb + 1), lb = ef_width(xb_last, nb + 1);
    H[H_MAGIC] = kMagic;
    H[H_N] = n;
    H[H_LEAF] = d.leaf | (static_cast<uint64_t>(class_extra[d.cls]) << 8);
    H[H_BUCKET] = in[i].bucket_size;
    H[H_NB] = nb;
    H[H_TBITS] = T_bits;
    H[H_MMAX] = h_set_max[i];
    H[H_BETA] = beta;
    H[H_DELTA_A] = static_cast<uint64_t>(delta_a);
    H[H_DELTA_B] = static_cast<uint64_t>(delta_b);
    H[H_LOW_A] = la;
    H[H_LOW_B] = lb;
    H[H_UP_A] = (xa_last >> la) + nb + 1;
    H[H_UP_B] = (xb_last >> lb) + nb + 1;
    layouts[i] = layout_of(H);
    H[H_WORDS] = layouts[i].total;
    H[H_CODES] = h_codes[i];
    blob_off[i + 1] = blob_off[i] + ((layouts[i].total + 31) & ~uint64_t(31));
    DevOut& o = houts[i];
    o.beta = beta;
    o.delta_a = delta_a;
    o.delta_b = delta_b;
    o.low_a = la;
    o.low_b = lb;
  }
  auto arena = std::make_shared<DeviceMem>();
  if ((rc = pool_alloc(&arena->p, blob_off[count] * sizeof(uint64_t), s))) return rc;
  uint64_t* d_arena = static_cast<uint64_t*>(arena->p);
  for (uint32_t i = 0; i < count; i++) {
    uint64_t* blob = d_arena + blob_off[i];
    DevOut& o = houts[i];
    o.blob = blob;
    std::copy_n(headers.data() + uint64_t(i) * kHeaderWords, kHeaderWords, o.header);
    o.tree = blob + layouts[i].tree;
    o.lower = blob + layouts[i].lower;
    o.upper_a = blob + layouts[i].upper_a;
    o.upper_b = blob + layouts[i].upper_b;
    o.anchors = blob + layouts[i].anchors;
    o.subs = reinterpret_cast<uint16_t*>(blob + layouts[i].subs);
  }
  RS_CUDA(cudaMemsetAsync(d_arena, 0, blob_off[count] * sizeof(uint64_t), s));
  RS_CUDA(cudaMemcpyAsync(d_outs, houts.data(), count * sizeof(DevOut), cudaMemcpyHostToDevice, s));

  // A6: Golomb-Rice codes; A7: Elias-Fano
  if (NB) {
    k_write_codes<<<grid_for(lanes), kBlock, 0, s>>>(counts, cbase, seeds, sizes, d_sets, count, d_outs, ct, off);
    count_launch();
  }
  k_ef_write<<<static_cast<unsigned>(elem_tiles), kBlock, 0, s>>>(d_sets, count, d_outs, rstart, off);
  count_launch();
  timer.mark();
  unsigned long long* work = nullptr;
  if (count_work) {
    uint32_t* code_leaf;
    if ((rc = sc.alloc(&work, 6)) || (rc = sc.alloc(&code_leaf, K + 1))) return rc;
    RS_CUDA(cudaMemsetAsync(work, 0, 6 * sizeof(unsigned long long), s));
    if (NB) {
      k_code_leaf<<<grid_for(NB), kBlock, 0, s>>>(cbase, bset, d_sets, NB, code_leaf);
      k_work<<<std::min<unsigned>(grid_for(K), sm_count * 8), kBlock, 0, s>>>(seeds, sizes, cbase + NB, code_leaf,
                                                                              work);
      count_launch(2);
    }
  }
  RS_CUDA(cudaGetLastError());
  unsigned long long w[6] = {0, 0, 0, 0, 0, 0}, x[2] = {0, 0};
  if (count_work) {
    RS_CUDA(cudaMemcpyAsync(w, work, sizeof(w), cudaMemcpyDeviceToHost, s));
    RS_CUDA(cudaMemcpyAsync(x, exec, sizeof(x), cudaMemcpyDeviceToHost, s));
  }
  RS_CUDA(cudaStreamSynchronize(s));

  for (uint32_t i = 0; i < count; i++) {
    Handle* h = new Handle();
    std::memcpy(h->header, headers.data() + uint64_t(i) * kHeaderWords, sizeof(h->header));
    h->layout = layouts[i];
    h->blob_mem = arena;
    h->table_mem = table_mem;
    h->d_blob = d_arena + blob_off[i];
    h->d_table = const_cast<uint64_t*>(ct.t[hs[i].cls]);
    h->table_mmax = ct.mmax[hs[i].cls];
    h->ncodes = h->header[H_CODES];
    h->range_size = h_R[i];
    h->device = dev;
    out[i] = h;
  }
  if (timer.on) {
    recsplit_profile_t pr{};
    pr.ms_signature = timer.ms(0, 1);
    pr.ms_group = timer.ms(1, 2);
    pr.ms_split = timer.ms(2, 3);
    pr.ms_leaf = timer.ms(3, 4);
    pr.ms_encode = timer.ms(4, 5);
    pr.ms_total = timer.ms(0, 5);
    pr.split_nodes = w[0];
    pr.split_trials = w[1];
    pr.split_evals = w[2];
    pr.leaf_nodes = w[3];
    pr.leaf_trials = w[4];
    pr.leaf_evals = w[5];
    pr.leaf_evals_executed = x[0];
    pr.split_evals_executed = x[1];
    pr.launches = launches_since(launch0);
    pr.split_levels = split_levels;
    store_profile(pr);
  }
  return RECSPLIT_OK;
}

// The searches' arguments hold kMaxClasses classes, and there are more pairs of
// leaf size and leaf range extra than that: sets of more classes are built in
// passes of kMaxClasses classes, in the order in which the classes first occur.
int build_sets(const SetInput* in, uint32_t count, const BuildOptions& opt, cudaStream_t s, Handle** out) {
  const double t_call = steady_ms();
  std::map<uint32_t, uint32_t> class_of;
  uint64_t keys = 0;
  for (uint32_t i = 0; i < count; i++) {
    out[i] = nullptr;
    if (in[i].leaf_extra > 32 - in[i].leaf) return fail(RECSPLIT_E_INVALID, "leaf size + leaf range extra above 32");
    class_of.emplace(class_key(in[i]), static_cast<uint32_t>(class_of.size()));
    keys += in[i].keys.n;
  }
  if (keys >= (1ull << 32)) return fail(RECSPLIT_E_INVALID, "at most 2^32 - 1 keys per build");
  if (count == 0) return RECSPLIT_OK;
  if (class_of.size() <= size_t(kMaxClasses)) return build_pass(in, count, opt, s, t_call, out);
  recsplit_profile_t sum{};
  for (uint32_t first = 0; first < class_of.size(); first += kMaxClasses) {
    std::vector<SetInput> sets;
    std::vector<uint32_t> at;
    for (uint32_t i = 0; i < count; i++)
      if (class_of[class_key(in[i])] - first < uint32_t(kMaxClasses)) {
        sets.push_back(in[i]);
        at.push_back(i);
      }
    std::vector<Handle*> built(sets.size(), nullptr);
    const int rc = build_pass(sets.data(), static_cast<uint32_t>(sets.size()), opt, s, t_call, built.data());
    for (size_t k = 0; k < at.size(); k++) out[at[k]] = built[k];
    if (rc) {
      for (uint32_t i = 0; i < count; i++) {
        delete out[i];
        out[i] = nullptr;
      }
      return rc;
    }
    recsplit_profile_t p;
    if (profiling_enabled() && !recsplit_last_profile(&p)) add_profile(&sum, p);
  }
  if (profiling_enabled()) store_profile(sum);
  return RECSPLIT_OK;
}

}  // namespace rs
