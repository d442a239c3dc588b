// Brute-force searches of Sec. 4: for every split node the first function
// index whose values send exactly k_t keys into the t-th interval of [0, m)
// (Sec. 5.1), and for every leaf the first index that maps the leaf's keys
// onto [0, m) (Sec. 5.2).
//
// Work unit of the light nodes: one node, searched by a group of G warps (G = 1, 2,
// 4 or 8 of the 8 warps of a CTA).  Lane L of warp w of a group tests indices
// w*32 + L, w*32 + L + 32G, ...; a warp stops after the round in which one of
// its lanes succeeds, or as soon as the group's best success so far is below
// its next round.  Every index below the final minimum has then been tested
// by its owner, so the group minimum is the first successful index (the
// result is deterministic and independent of G).  Nodes are handed out by an
// atomic counter (persistent CTAs), in larger groups where there are fewer nodes
// than warps.  Leaves of 4 to 8 keys share a warp four at a time
// (k_leaves_packed); heavy split nodes and leaves of 13 keys or more are
// searched by all CTAs that would otherwise idle (shared_nodes).
//
// What bounds the searches: an evaluation of the hash family alone takes 20.5 to
// 21.5 cycles per warp and sub-partition (six 32-bit multiplies on one pipe, seven
// shifts and xors on the other; occupancy, uniform registers and other forms of the
// products made no difference), so a search's floor is its evaluations times
// that, and what it adds per evaluation is kept to the counting of one value.
#include <algorithm>
#include <array>
#include <climits>
#include <mutex>
#include <utility>

#include "device.cuh"

namespace rs {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ void group_sync(uint32_t gid, uint32_t gwarps) {
  if (gwarps == 1) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(gid + 1), "r"(gwarps * 32) : "memory");
  }
}

__device__ __forceinline__ uint64_t shl64(uint64_t x, uint32_t s) {
  uint64_t r;  // PTX clamps shift amounts above 64 to 64 (result 0)
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
}
__device__ __forceinline__ uint32_t shl32(uint32_t x, uint32_t s) {
  uint32_t r;  // clamps above 32 (result 0)
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
}

__device__ __forceinline__ void set_error(int* err, int code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ uint64_t volatile_load(const uint64_t* p) {
  return *reinterpret_cast<const volatile uint64_t*>(p);
}

// Stall threshold: a node that has not succeeded after 64 times its expected
// number of trials (probability about e^-64) is checked for keys that can
// never be separated.
__device__ __forceinline__ uint64_t stall_threshold(const uint64_t* table, uint32_t m) {
  const uint64_t e = table[kTableWords * m + 2];
  return e > (kMaxTrials >> 6) ? kMaxTrials : e << 6;
}

// Trial limit of a node: 2^36, or 1024 times its expected number of trials
// (at least 4096) if that is smaller.  A correct search passes it with
// probability below e^-1024; the limit bounds the time of a search that can
// never succeed.
__device__ __forceinline__ uint64_t trial_limit(const uint64_t* table, uint32_t m) {
  const uint64_t e = table[kTableWords * m + 2];
  if (e > (kMaxTrials >> 10)) return kMaxTrials;
  return max(uint64_t(4096), e << 10);
}

// ---------------------------------------------------------------- split trial
// Part t of a key is floor(phi / unit) (at most fanout - 1).  Counts of the
// first fanout - 1 parts are packed in fields of B bits (2^B > m, so no field
// overflows); success iff the packed sum equals the packed target.
//
// For fanouts of at most 3 the parts are not computed.  With h the top 32
// bits of the hash, phi = floor(h * m / 2^32) < k * unit holds exactly when
// h < T_k = ceil(k * unit * 2^32 / m) (T_k < 2^32 because k * unit < m), so
// the split is the one sought iff m - k * unit keys have h >= T_k for k = 1 ..
// fanout - 1.  This replaces two multiply-highs and a variable shift per key
// by fanout - 1 additions with carry.
// Largest fanout searched by thresholds: with three thresholds (fanout 4) the
// compares cost about as much as the multiply-highs they replace.
constexpr uint32_t kMaxThresholdFanout = 3;

struct SplitParams {
  uint32_t m, unit, fanout, bits, magic;  // magic = ceil(2^32 / unit): exact for m < 2^16, unit >= 2
  uint64_t target, mask;
  uint32_t thr1, thr2;      // T_1, T_2 (threshold modes)
  uint32_t nbits, nmask, ntarget;  // narrow fields (modes 5, 7): 2^nbits > unit
  bool confirm;                    // mode 7: fields can overflow, confirm matches exactly
  const uint32_t* sets;            // modes 8, 9: packed counts of four parts (fill_part_counts)
  uint32_t tail;                   // modes 8, 9 on shared nodes: keys of the second phase
};

// Modes 8 and 9: F = 5 .. 7 equal parts (m = F unit).  The part of a key, 3
// bits, is the top of floor(F 2^29 h / 2^32); the parts of four keys are
// shifted into one 12-bit word (one funnel shift per key, where counting a
// part takes a shift-and-add, a shift and an add), and a table of 4096 words in
// shared memory gives their counts in fields: 6 fields of 5 bits (mode 8: unit <
// 32) or 4 of 8 bits (mode 9: F = 5, unit < 256).  The last part is implied.
constexpr uint32_t kPartCounts = 4096;

__device__ __forceinline__ uint32_t part_one(uint32_t part, uint32_t bits, uint32_t fields) {
  return part < fields ? 1u << (part * bits) : 0u;
}

// The two tables, 5-bit fields then 8-bit fields, from those of two parts
// (called by the whole CTA).
__device__ __forceinline__ void fill_part_counts(uint32_t* t) {
  __shared__ uint32_t two[2][64];
  if (threadIdx.x < 64) {
    const uint32_t p = threadIdx.x & 7, q = threadIdx.x >> 3;
    two[0][threadIdx.x] = part_one(p, 5, 6) + part_one(q, 5, 6);
    two[1][threadIdx.x] = part_one(p, 8, 4) + part_one(q, 8, 4);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < kPartCounts; i += kThreads) {
    t[i] = two[0][i >> 6] + two[0][i & 63];
    t[kPartCounts + i] = two[1][i >> 6] + two[1][i & 63];
  }
  __syncthreads();
}

// MODE 0: 32-bit fields + magic; 1: 64-bit fields + magic; 2: 64-bit +
// division; 3, 4: thresholds for fanout 2, 3;
// 5: 32-bit fields of nbits bits (2^nbits > unit but possibly <= m) + magic.
// In mode 5 a field can overflow into the next one, so a match may be false,
// but never missed: when every counted part has exactly unit keys no field
// overflows.  A match is confirmed with the exact 64-bit count (mode 1).
// 6: four parts of equal size (m = 4 unit < 256): the part is
// floor(floor(h m / 2^32) / unit) = floor(4 h / 2^32), the top two bits of h.
// 7: F parts of equal size (m = F unit): the part is floor(F h / 2^32), one
// multiply-high instead of two, counted in nbits-bit fields; when a field
// can overflow (2^nbits <= m) a match is confirmed exactly as in mode 5.
// 8, 9: mode 7 with fields of 5 and 8 bits by table (above).
// Modes 3 and 4: c1 and c2 count the keys with h >= T_1 and h >= T_2, the carry
// of h + (2^32 - T) added by add-with-carry.  These two additions issue to
// either pipe (1.4 cycles per warp together); a compare and a predicated
// add take 2.2.
template <int MODE>
__device__ __forceinline__ void count_thresholds(uint32_t h, const SplitParams& p, uint32_t& c1, uint32_t& c2) {
  asm("{.reg .u32 t; add.cc.u32 t, %1, %2; addc.u32 %0, %0, 0;}" : "+r"(c1) : "r"(h), "r"(0u - p.thr1));
  if (MODE == 4) asm("{.reg .u32 t; add.cc.u32 t, %1, %2; addc.u32 %0, %0, 0;}" : "+r"(c2) : "r"(h), "r"(0u - p.thr2));
}

template <int MODE>
__device__ __forceinline__ bool threshold_match(const SplitParams& p, uint32_t c1, uint32_t c2) {
  return c1 == p.m - p.unit && (MODE == 3 || c2 == p.m - 2 * p.unit);
}

template <bool STAGED>
__device__ __forceinline__ ulonglong2 key_pair(const uint64_t* keys) {
  if (STAGED) return *reinterpret_cast<const ulonglong2*>(keys);
  return make_ulonglong2(keys[0], keys[1]);
}

// Fields of modes 8 and 9 of keys [j0, j1) under function kp, j0 even.
template <int MODE, bool STAGED>
__device__ __forceinline__ uint32_t split_fields(const uint64_t* __restrict__ keys, const SplitParams& p, uint64_t kp,
                                                 uint32_t j0, uint32_t j1) {
  constexpr uint32_t kBits = MODE == 8 ? 5 : 8, kFields = MODE == 8 ? 6 : 4;
  const uint32_t scale = p.fanout << 29;
  uint32_t acc = 0, j = j0;
#pragma unroll 2
  for (; j + 4 <= j1; j += 4) {
    const ulonglong2 x = key_pair<STAGED>(keys + j), y = key_pair<STAGED>(keys + j + 2);
    uint32_t v = __umulhi(family_top32(x.x, kp), scale) >> 29;
    v = __funnelshift_l(__umulhi(family_top32(x.y, kp), scale), v, 3);
    v = __funnelshift_l(__umulhi(family_top32(y.x, kp), scale), v, 3);
    v = __funnelshift_l(__umulhi(family_top32(y.y, kp), scale), v, 3);
    acc += p.sets[v];
  }
#pragma unroll 1
  for (; j < j1; j++) acc += part_one(__umulhi(family_top32(keys[j], kp), p.fanout), kBits, kFields);
  return acc;
}

// STAGED: the keys are in shared memory, 16-byte aligned: modes 3, 4, 6, 8 and
// 9 read them two at a time.
template <int MODE, bool STAGED>
__device__ __forceinline__ bool split_trial(const uint64_t* __restrict__ keys, const SplitParams& p,
                                            uint64_t kp) {
  if constexpr (MODE >= 8) {
    return (split_fields<MODE, STAGED>(keys, p, kp, 0, p.m) & p.nmask) == p.ntarget;
  } else if (MODE == 6) {
    // the two-bit parts are shifted into words of 16 keys (one funnel shift
    // per key, where counting fields takes four instructions), and the parts
    // 1, 2 and 3 are counted with population counts; part 0 is implied
    uint32_t low = 0, high = 0, both = 0;
    uint32_t j = 0;
#pragma unroll 1
    for (; j + 16 <= p.m; j += 16) {
      uint32_t w = 0;
#pragma unroll
      for (uint32_t t = 0; t < 16; t += 2) {
        const ulonglong2 x = key_pair<STAGED>(keys + j + t);
        w = __funnelshift_l(family_top32(x.x, kp), w, 2);
        w = __funnelshift_l(family_top32(x.y, kp), w, 2);
      }
      low += __popc(w & 0x55555555u);
      high += __popc(w & 0xAAAAAAAAu);
      both += __popc(w & (w >> 1) & 0x55555555u);
    }
    if (j < p.m) {
      uint32_t w = 0;
#pragma unroll 4
      for (; j < p.m; j++) w = __funnelshift_l(family_top32(keys[j], kp), w, 2);
      low += __popc(w & 0x55555555u);
      high += __popc(w & 0xAAAAAAAAu);
      both += __popc(w & (w >> 1) & 0x55555555u);
    }
    return low == 2 * p.unit && high == 2 * p.unit && both == p.unit;
  } else if (MODE == 7) {
    uint32_t acc = 0;
#pragma unroll 4
    for (uint32_t j = 0; j < p.m; j++) acc += shl32(1u, __umulhi(family_top32(keys[j], kp), p.fanout) * p.nbits);
    return (acc & p.nmask) == p.ntarget;
  } else if (MODE == 3 || MODE == 4) {
    uint32_t c1 = 0, c2 = 0, j = 0;
#pragma unroll 1
    for (; j + 8 <= p.m; j += 8) {
#pragma unroll
      for (uint32_t t = 0; t < 8; t += 2) {
        const ulonglong2 x = key_pair<STAGED>(keys + j + t);
        count_thresholds<MODE>(family_top32(x.x, kp), p, c1, c2);
        count_thresholds<MODE>(family_top32(x.y, kp), p, c1, c2);
      }
    }
#pragma unroll 1
    for (; j < p.m; j++) count_thresholds<MODE>(family_top32(keys[j], kp), p, c1, c2);
    return threshold_match<MODE>(p, c1, c2);
  } else if (MODE == 0) {
    uint32_t acc = 0;
#pragma unroll 4
    for (uint32_t j = 0; j < p.m; j++) {
      const uint32_t v = phi_pre(keys[j], kp, p.m);
      acc += shl32(1u, __umulhi(v, p.magic) * p.bits);
    }
    return (acc & static_cast<uint32_t>(p.mask)) == static_cast<uint32_t>(p.target);
  } else if (MODE == 5) {
    uint32_t acc = 0;
#pragma unroll 4
    for (uint32_t j = 0; j < p.m; j++) {
      const uint32_t v = phi_pre(keys[j], kp, p.m);
      acc += shl32(1u, __umulhi(v, p.magic) * p.nbits);
    }
    return (acc & p.nmask) == p.ntarget;
  } else {
    uint64_t acc = 0;
#pragma unroll 4
    for (uint32_t j = 0; j < p.m; j++) {
      const uint32_t v = phi_pre(keys[j], kp, p.m);
      const uint32_t part = MODE == 1 ? __umulhi(v, p.magic) : min(v / p.unit, p.fanout - 1);
      acc += shl64(1ull, part * p.bits);
    }
    return (acc & p.mask) == p.target;
  }
}

// Any two equal keys (they can never be separated)?  Lanes split the pairs.
__device__ bool has_duplicate(const uint64_t* keys, uint32_t m, uint32_t lane) {
  bool dup = false;
  for (uint32_t i = lane; i < m && !dup; i += 32) {
    const uint64_t x = keys[i];
    for (uint32_t j = i + 1; j < m; j++)
      if (keys[j] == x) {
        dup = true;
        break;
      }
  }
  return __any_sync(0xFFFFFFFFu, dup);
}

template <int MODE, bool STAGED>
__device__ __forceinline__ void split_search_warp(const uint64_t* __restrict__ keys, const SplitParams& sp,
                                                  uint32_t depth, uint32_t wig, uint32_t gwarps, uint32_t lane,
                                                  uint64_t* best, uint64_t stall, uint64_t limit,
                                                  int* err, unsigned long long* exec) {
  bool checked = false;
  uint32_t rounds = 0;
  for (uint64_t base = uint64_t(wig) * 32;; base += uint64_t(gwarps) * 32) {
    if (gwarps > 1 && __any_sync(0xFFFFFFFFu, base >= volatile_load(best))) break;
    if ((++rounds & 255) == 0 && __shfl_sync(0xFFFFFFFFu, lane == 0 ? *reinterpret_cast<volatile int*>(err) : 0, 0))
      break;  // another search failed, or the host cancelled the build
    if (base >= limit) {
      if (lane == 0) {
        set_error(err, RECSPLIT_E_SEARCH_LIMIT);
        atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
      }
      break;
    }
    if (!checked && base >= stall) {
      checked = true;
      if (has_duplicate(keys, sp.m, lane)) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_DUPLICATE);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        break;
      }
    }
    const uint64_t kp = family_key(base + lane, depth);
    bool ok = split_trial<MODE, STAGED>(keys, sp, kp);
    if ((MODE == 5 || (MODE >= 7 && sp.confirm)) && ok) ok = split_trial<1, STAGED>(keys, sp, kp);
    const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
    if (exec && lane == 0) *exec += 32 * sp.m;
    if (hits) {
      if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), base + __ffs(hits) - 1);
      break;
    }
  }
}

// Threshold nodes that take few trials (a binary split of 100 keys with 96 on
// one side takes 5): a round of 32 indices is mostly wasted, so four lanes
// share an index, each counting every fourth key, and a round tests 8.  It
// saves about 12 of 32 indices per node and costs about 25 instructions per
// round more (m/4 keys of about 15 instructions each), which pays while the
// expected trials stay below the node's keys.
template <int MODE>
__device__ __forceinline__ void split_search_few(const uint64_t* __restrict__ keys, const SplitParams& sp,
                                                 uint32_t depth, uint32_t wig, uint32_t gwarps, uint32_t lane,
                                                 uint64_t* best, uint64_t stall, uint64_t limit, int* err,
                                                 unsigned long long* exec) {
  bool checked = false;
  uint32_t rounds = 0;
  for (uint64_t base = uint64_t(wig) * 8;; base += uint64_t(gwarps) * 8) {
    if (gwarps > 1 && __any_sync(0xFFFFFFFFu, base >= volatile_load(best))) break;
    if ((++rounds & 255) == 0 && __shfl_sync(0xFFFFFFFFu, lane == 0 ? *reinterpret_cast<volatile int*>(err) : 0, 0))
      break;  // another search failed, or the host cancelled the build
    if (base >= limit) {
      if (lane == 0) {
        set_error(err, RECSPLIT_E_SEARCH_LIMIT);
        atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
      }
      break;
    }
    if (!checked && base >= stall) {
      checked = true;
      if (has_duplicate(keys, sp.m, lane)) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_DUPLICATE);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        break;
      }
    }
    const uint64_t kp = family_key(base + (lane >> 2), depth);
    uint32_t c1 = 0, c2 = 0;
#pragma unroll 4
    for (uint32_t j = lane & 3; j < sp.m; j += 4) count_thresholds<MODE>(family_top32(keys[j], kp), sp, c1, c2);
    uint32_t c = MODE == 4 ? c1 | (c2 << 16) : c1;  // counts below 2^16
    c += __shfl_xor_sync(0xFFFFFFFFu, c, 1);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, 2);
    const bool ok = threshold_match<MODE>(sp, MODE == 4 ? c & 0xFFFFu : c, c >> 16);
    const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
    if (exec && lane == 0) *exec += 8 * sp.m;
    if (hits) {
      if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), base + ((__ffs(hits) - 1) >> 2));
      break;
    }
  }
}

// A node too large to be staged (more than 1536 keys) has more keys than the
// upper unit of any leaf size (1296 at l = 24), so it is split in two: modes 3
// and 2 are all it needs.
template <bool STAGED>
__device__ __forceinline__ void split_search(const uint64_t* __restrict__ keys, const SplitParams& sp, int mode,
                                             uint32_t depth, uint32_t wig, uint32_t gwarps, uint32_t lane,
                                             uint64_t* best, uint64_t stall, uint64_t limit, int* err,
                                             unsigned long long* exec) {
  if (STAGED) {
    if (stall <= uint64_t(sp.m) << 6) {  // stall = 64 times the expected trials
      if (mode == 3) return split_search_few<3>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      if (mode == 4) return split_search_few<4>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
    }
    switch (mode) {
      case 0: return split_search_warp<0, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 1: return split_search_warp<1, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 4: return split_search_warp<4, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 5: return split_search_warp<5, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 6: return split_search_warp<6, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 7: return split_search_warp<7, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 8: return split_search_warp<8, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
      case 9: return split_search_warp<9, true>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
    }
  }
  if (mode == 3)
    split_search_warp<3, STAGED>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
  else
    split_search_warp<2, STAGED>(keys, sp, depth, wig, gwarps, lane, best, stall, limit, err, exec);
}

// Emits the children of a split node with at least two keys into the queues
// of full leaves, partial leaves or next-level splits, light or heavy (one
// warp).
__device__ void emit_children(const SearchArgs& a, const Node& nd, const uint64_t* table, uint64_t w1, uint32_t leaf,
                              uint32_t lane) {
  const uint32_t unit = static_cast<uint32_t>(w1), fanout = static_cast<uint32_t>(w1 >> 32) & 0xFF;
  const uint32_t t = lane;
  const uint32_t k = t + 1 < fanout ? unit : nd.m - unit * (fanout - 1);
  const bool valid = t < fanout && k >= 2;
  const uint32_t kind =
      !valid ? 4 : (k == leaf ? 0 : (k < leaf ? 1 : (heavy_flag(w1, t + 1 < fanout ? 1 : 2, a.heavy_flag) ? 3 : 2)));
  const uint32_t c_of_node = nd.depth >> 8;
  const uint32_t unit_codes = static_cast<uint32_t>(table[kTableWords * unit] >> 32);
  Node child;
  child.start = nd.start + t * unit;
  child.m = k;
  child.slot = nd.slot + 1 + t * unit_codes;
  child.depth = nd.depth + 1;
#pragma unroll
  for (uint32_t c = 0; c < 4; c++) {
    const bool mine = kind == c;
    const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, mine);
    if (!ballot) continue;
    const uint32_t leader = __ffs(ballot) - 1;
    Node* q = c == 0 ? a.full_q[c_of_node] : (c == 1 ? a.part_q[c_of_node] : a.split_out[c - 2]);
    uint32_t* cnt = c == 0 ? a.full_n + c_of_node : (c == 1 ? a.part_n + c_of_node : a.split_out_count[c - 2]);
    const uint32_t cap = c == 0 ? a.full_cap[c_of_node] : (c == 1 ? a.part_cap[c_of_node] : a.split_cap[c - 2]);
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(ballot));
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    const uint32_t at = base + __popc(ballot & ((1u << lane) - 1));
    if (mine) {
      if (at < cap)
        q[at] = child;
      else
        set_error(a.error, RECSPLIT_E_INVALID);  // a queue would overflow: never for correct sizes
    }
  }
}

// Search parameters of a split node; returns the count mode (split_trial).
// counts: the tables of modes 8 and 9, or null if the launch has none.
__device__ __forceinline__ int split_setup(const Node& nd, const uint64_t* table, const uint32_t* counts,
                                           SplitParams& sp) {
  const uint64_t w1 = table[kTableWords * nd.m + 1];
  sp.m = nd.m;
  sp.unit = static_cast<uint32_t>(w1);
  sp.fanout = static_cast<uint32_t>(w1 >> 32) & 0xFF;
  sp.bits = 32 - __clz(nd.m);
  // ceil(2^32 / unit), from the table (word 3): stored where the
  // multiply-high gives floor(v / unit) for every v < m (always for m < 2^16
  // and unit >= 2), else 0, and the search divides
  sp.magic = static_cast<uint32_t>(table[kTableWords * nd.m + 3]);
  const uint32_t fields = sp.fanout - 1;
  sp.target = 0;
  for (uint32_t t = 0; t < fields; t++) sp.target |= uint64_t(sp.unit) << (t * sp.bits);
  sp.mask = fields * sp.bits >= 64 ? ~0ull : (1ull << (fields * sp.bits)) - 1;
  int mode = (nd.m >= 65536 || sp.unit < 2 || sp.magic == 0) ? 2 : (fields * sp.bits <= 32 ? 0 : 1);
  if (sp.fanout == 4 && nd.m == 4 * sp.unit && nd.m < 256) {
    mode = 6;
  } else if (sp.fanout >= 5 && nd.m == sp.fanout * sp.unit && sp.unit >= 2 && nd.m < 65536) {
    uint32_t nb = nd.m < 256 && fields * 8 <= 32 ? 8 : 32 - __clz(sp.unit);
    if (counts && sp.fanout == 5 && sp.unit < 256)
      mode = 9, nb = 8;
    else if (counts && sp.fanout <= 7 && sp.unit < 32)
      mode = 8, nb = 5;
    if (fields * nb <= 32) {
      if (mode >= 8) {
        sp.sets = counts + (mode == 8 ? 0 : kPartCounts);
        // second-phase keys of the two-phase block search (speed only: any
        // value from 1 to m - 1 gives the same index); about 1.75 sqrt(m)
        // minimises the modelled work (19 of 112 keys, 18 of 96, 42 of 560),
        // with whole fours in the first phase; below 90 keys too many indices
        // reach the second phase (three of five at 60 keys)
        const uint32_t head = nd.m - static_cast<uint32_t>(1.75f * sqrtf(static_cast<float>(nd.m))) - 1;
        sp.tail = nd.m < 90 ? 0 : nd.m - (head & ~3u);
      } else {
        mode = 7;
      }
      sp.confirm = (1u << nb) <= nd.m;
      sp.nbits = nb;
      sp.nmask = fields * nb == 32 ? ~0u : (1u << (fields * nb)) - 1;
      sp.ntarget = 0;
      for (uint32_t t = 0; t < fields; t++) sp.ntarget |= sp.unit << (t * nb);
    }
  }
  if (mode == 1 && sp.fanout * sp.unit != nd.m) {
    sp.nbits = 32 - __clz(sp.unit);
    if (fields * sp.nbits <= 32) {
      mode = 5;
      sp.nmask = fields * sp.nbits == 32 ? ~0u : (1u << (fields * sp.nbits)) - 1;
      sp.ntarget = 0;
      for (uint32_t t = 0; t < fields; t++) sp.ntarget |= sp.unit << (t * sp.nbits);
    }
  }
  if (nd.m < 65536 && sp.fanout >= 2 && sp.fanout <= kMaxThresholdFanout && fields * sp.bits <= 32) {
    mode = 1 + static_cast<int>(sp.fanout);
    // T_k = ceil(k * unit * 2^32 / m), k = 1 on even lanes and 2 on odd ones, in
    // two 16-bit digits (32-bit divisions: m < 2^16, and k * unit < m where T_k
    // is used)
    const uint32_t u = sp.unit << (threadIdx.x & 1);
    const uint32_t q1 = (u << 16) / nd.m, r1 = (u << 16) % nd.m;
    const uint32_t q0 = (r1 << 16) / nd.m, r0 = (r1 << 16) % nd.m;
    const uint32_t thr = (q1 << 16) + q0 + (r0 ? 1u : 0u);
    sp.thr1 = __shfl_sync(0xFFFFFFFFu, thr, 0);
    sp.thr2 = __shfl_sync(0xFFFFFFFFu, thr, 1);
  }
  return mode;
}

// Stores the node's index and partitions its keys with it into the
// children's ranges of the other key array, then queues the children (the
// threads tig < gthreads of one group; `fill` is the group's 16 part cursors,
// zero on entry; `mine` the node's keys if staged, else null).
__device__ __forceinline__ void partition_node(const SearchArgs& a, const Node& nd, uint64_t seed,
                                               const uint64_t* mine, uint32_t tig, uint32_t gthreads, uint32_t lane,
                                               bool first_warp, uint32_t* fill) {
  const uint32_t cls = nd.depth >> 8, depth = nd.depth & kDepthMask;
  const uint64_t* table = a.table[cls];
  const uint64_t w1 = table[kTableWords * nd.m + 1];
  const uint32_t unit = static_cast<uint32_t>(w1), fanout = static_cast<uint32_t>(w1 >> 32) & 0xFF;
  const uint32_t magic = static_cast<uint32_t>(table[kTableWords * nd.m + 3]);  // ceil(2^32 / unit) or 0
  const bool divide = nd.m >= 65536 || unit < 2 || magic == 0;
  const uint64_t* src = a.keys[depth & 1] + nd.start;
  uint64_t* dst = a.keys[(depth + 1) & 1] + nd.start;
  if (tig == 0) {
    a.seeds[nd.slot] = seed;
    a.sizes[nd.slot] = nd.m;
  }
  const uint64_t kp = family_key(seed, depth);
  const uint64_t* from = mine ? mine : src;
  for (uint32_t j = tig; j < nd.m; j += gthreads) {
    const uint64_t x = from[j];
    const uint32_t v = phi_pre(x, kp, nd.m);
    const uint32_t part = min(divide ? v / unit : __umulhi(v, magic), fanout - 1);
    const uint32_t pos = atomicAdd(&fill[part], 1u);
    const uint32_t at = part * unit + pos;
    if (at < nd.m)
      dst[at] = x;
    else
      set_error(a.error, RECSPLIT_E_INVALID);  // unreachable for a correct split
  }
  if (first_warp) emit_children(a, nd, table, w1, a.leaf_of[cls], lane);
}

// Warps per node or leaf: the launch shape's, doubled (up to the CTA) while
// the launch then has at most `spread` groups' worth of work items for the
// warps of the grid.  Their number is known on the device only.  A launch of
// few items lasts as long as its longest search, so more warps on each help:
// split and leaf phases at l = 8, b = 100: 10^3 keys 87 + 69 -> 47 + 21 us, 10^5
// keys 197 + 85 -> 97 + 75 us; l = 10, b = 100, 3 * 10^5 keys 241 -> 179 us (split,
// spread 4 against 1).  spread is 4 where a search takes several rounds of 32
// indices (128 trials) and 2 below, where four warps mostly test past the
// winner (l = 8, 10^5 keys: split 97 us with 2, 117 us with 4), and 32 where it
// takes long (2048 trials, leaves from l = 10; leaf phase, b = 100, spread 4, 16 and 32: l =
// 11, 10^5 keys 633, 559 and 561 us, 3 * 10^5 1719, 1539 and 1376, from 10^6 on equal; l = 12,
// 10^5 1184, 1114 and 1120; but l = 10, 10^5 260, 295 and 300, 3 * 10^5 655, 616 and 631).
__device__ __forceinline__ uint32_t group_warps(uint32_t gwarps, uint32_t items, uint32_t spread) {
  while (gwarps < kWarps && uint64_t(items) * gwarps * 2 <= spread * gridDim.x * kWarps) gwarps *= 2;
  return gwarps;
}
__host__ __device__ constexpr uint32_t group_spread(uint64_t trials) {
  return trials >= 2048 ? 32 : (trials >= 128 ? 4 : 2);
}

// Light split nodes of a level.  COUNT: work counting (the evaluations executed go to a.exec_count[1]);
// without it the counter is compiled out.
template <bool COUNT>
__global__ void __launch_bounds__(kThreads, 4) k_split_level(SearchArgs a, uint32_t gwarps, uint32_t cap,
                                                             uint32_t tables, uint32_t spread) {
  extern __shared__ __align__(16) uint64_t dynamic[];  // tables of modes 8 and 9 if any, then the groups' keys
  __shared__ uint64_t best[kWarps];
  __shared__ uint32_t task[kWarps];
  __shared__ uint32_t fill[kWarps][16];
  __shared__ unsigned long long wexec[kWarps];  // work counting: evaluations per warp, flushed at exit
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (COUNT && lane == 0) wexec[warp] = 0;
  const uint32_t total = *a.split_in_count[0];
  // (a counting build keeps the launch shape: with one warp per node its count is
  // the same in every build)
  if (!COUNT) gwarps = group_warps(gwarps, total, spread);
  const uint32_t gid = warp / gwarps, wig = warp % gwarps;
  const uint32_t tig = wig * 32 + lane, gthreads = gwarps * 32;
  const bool leader = wig == 0 && lane == 0;
  const uint32_t* const counts = tables ? reinterpret_cast<const uint32_t*>(dynamic) : nullptr;
  if (tables) fill_part_counts(reinterpret_cast<uint32_t*>(dynamic));
  uint64_t* mine = dynamic + (tables ? kPartCounts : 0) + size_t(gid) * cap;

  for (;;) {
    if (leader) task[gid] = *reinterpret_cast<volatile int*>(a.error) ? total : atomicAdd(a.work_counter, 1u);
    group_sync(gid, gwarps);
    const uint32_t idx = task[gid];
    if (idx >= total) break;
    {
      // search: the parameters live only for this scope, so the registers
      // of the search loops are not shared with the partition step's state
      const Node nd = a.split_in[0][idx];
      const uint32_t depth = nd.depth & kDepthMask;
      const uint64_t* table = a.table[nd.depth >> 8];
      SplitParams sp;
      const int mode = split_setup(nd, table, counts, sp);
      const uint64_t stall = stall_threshold(table, nd.m);
      const uint64_t limit = trial_limit(table, nd.m);

      const uint64_t* src = a.keys[depth & 1] + nd.start;
      const bool in_smem = nd.m <= cap;
      if (in_smem)
        for (uint32_t j = tig; j < nd.m; j += gthreads) mine[j] = src[j];
      if (leader) best[gid] = ~0ull;
      if (tig < 16) fill[gid][tig] = 0;
      group_sync(gid, gwarps);

      unsigned long long* exec = COUNT ? &wexec[warp] : nullptr;
      if (in_smem)
        split_search<true>(mine, sp, mode, depth, wig, gwarps, lane, &best[gid], stall, limit, a.error, exec);
      else
        split_search<false>(src, sp, mode, depth, wig, gwarps, lane, &best[gid], stall, limit, a.error, exec);
      group_sync(gid, gwarps);
    }

    const uint64_t seed = best[gid];
    if (!*reinterpret_cast<volatile int*>(a.error)) {
      const Node nd = a.split_in[0][idx];
      partition_node(a, nd, seed, nd.m <= cap ? mine : nullptr, tig, gthreads, lane, wig == 0, fill[gid]);
    }
    group_sync(gid, gwarps);
  }
  if (COUNT && lane == 0 && wexec[warp]) atomicAdd(a.exec_count + 1, wexec[warp]);
}

// ---------------------------------------------------------------- shared nodes
// Levels whose nodes each need many trials (a node's expected work of
// trials x keys is large, e.g. the 560 -> 5 x 112 and 112 -> 7 x 16 splits at
// l = 16, b = 2000) end on a few long searches: trial counts are geometric,
// so while the last nodes run, the CTAs that found the queue empty would sit
// idle.  On these levels a CTA that finds the queue empty joins a node still
// in progress instead.  Every participant's warps claim blocks of
// kShareRounds * 32 consecutive indices from the node's block counter and
// test them in order; a warp stops at its first success (atomicMin into the
// node's best) or at a block that starts at or above the best.  Blocks are
// claimed in increasing order, so every index below the final best was tested
// and the result is the first successful index, whatever the participants.
// The last participant to leave (refs drops to 0 and it closes the node)
// partitions the keys and queues the children.
constexpr uint32_t kShareRounds = 4;
constexpr uint32_t kMaxJoins = 4096;  // nodes one CTA may join in one launch

// Two-phase test of one claimed block (kShareRounds * 32 indices from base0)
// for the equal-part modes 8 and 9: phase 1 counts the first m - tail keys of
// every index and keeps, in index order, those whose parts all still hold at
// most unit keys; phase 2 adds the last tail keys of the survivors, 32 at a
// time, and applies the one-phase test to the sum (the same fields: the
// accumulation is a sum).  An index dropped in phase 1 has a part with more
// than unit keys, so the one-phase test (after its exact confirmation) would
// reject it too: the smallest successful index of the block is unchanged.
// While every part holds at most unit < 2^NB keys no field overflows, so the
// fields read in phase 1 are exact for the indices that are kept; an index
// whose fields overflowed has a part beyond unit and may be kept or dropped.
// Returns the evaluations executed; `hit` the smallest successful index, if any.
template <int MODE, bool STAGED>
__device__ __forceinline__ uint64_t shared_block_two_phase(const uint64_t* __restrict__ keys, const SplitParams& sp,
                                                           uint32_t depth, uint32_t lane, uint64_t base0,
                                                           uint64_t* best, uint4* surv, uint64_t* hit) {
  constexpr uint32_t NB = MODE == 8 ? 5 : 8;
  const uint32_t head = sp.m - sp.tail, fmask = (1u << NB) - 1;
  const uint32_t below = (1u << lane) - 1;
  uint64_t evals = 0;
  uint32_t ns = 0;
  for (uint32_t r = 0; r < kShareRounds; r++) {
    const uint64_t base = base0 + r * 32;
    if (r && base >= volatile_load(best)) break;  // a smaller index is known: the rest cannot win
    const uint64_t kp = family_key(base + lane, depth);
    const uint32_t acc = split_fields<MODE, STAGED>(keys, sp, kp, 0, head);
    uint32_t counted = 0;
    bool keep = true;
    for (uint32_t t = 0; t + 1 < sp.fanout; t++) {
      const uint32_t f = (acc >> (t * NB)) & fmask;
      keep &= f <= sp.unit;
      counted += f;
    }
    keep &= counted <= head && head - counted <= sp.unit;  // the last part
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, keep);
    if (keep)
      surv[ns + __popc(b & below)] =
          make_uint4(r * 32 + lane, acc, static_cast<uint32_t>(kp), static_cast<uint32_t>(kp >> 32));
    ns += __popc(b);
    evals += 32 * head;
  }
  __syncwarp();
  *hit = ~0ull;
  for (uint32_t t0 = 0; t0 < ns; t0 += 32) {
    const uint32_t t = t0 + lane;
    bool ok = false;
    if (t < ns) {
      const uint4 e = surv[t];
      const uint64_t kp = (uint64_t(e.w) << 32) | e.z;
      const uint32_t acc = e.y + split_fields<MODE, STAGED>(keys, sp, kp, head, sp.m);
      ok = (acc & sp.nmask) == sp.ntarget;
      if (ok && sp.confirm) ok = split_trial<1, STAGED>(keys, sp, kp);
    }
    evals += uint64_t(min(32u, ns - t0)) * sp.tail;
    const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
    if (hits) {
      *hit = base0 + surv[t0 + __ffs(hits) - 1].x;
      break;
    }
  }
  __syncwarp();
  return evals;
}

// Returns the evaluations the warp executed (32 * m per round of 32 indices,
// or as counted by the two-phase block test).
template <int MODE, bool STAGED>
__device__ __forceinline__ uint64_t shared_search_warp(const uint64_t* __restrict__ keys, const SplitParams& sp,
                                                       uint32_t depth, uint32_t lane, uint64_t* best,
                                                       unsigned int* next, uint64_t stall, uint64_t limit,
                                                       int* err, uint4* surv) {
  uint32_t blocks = 0;
  uint64_t evals = 0;
  for (;;) {
    uint32_t blk = 0;
    if (lane == 0) blk = atomicAdd(next, 1u);
    const uint64_t base0 = uint64_t(__shfl_sync(0xFFFFFFFFu, blk, 0)) * (kShareRounds * 32);
    if (base0 >= volatile_load(best)) return evals;
    if ((++blocks & 63) == 0 && __shfl_sync(0xFFFFFFFFu, lane == 0 ? *reinterpret_cast<volatile int*>(err) : 0, 0))
      return evals;  // another search failed, or the host cancelled the build
    // Blocks at or beyond the limit are not searched.  Participants claim
    // ahead of the frontier, so a claim there does not mean the search
    // failed: the node's closer reports the limit if no index below it
    // succeeded (every block below it was then claimed and tested).
    if (base0 >= limit) return evals;
    // the one warp whose block holds the stall point checks for keys that
    // can never be separated (an O(m^2) scan, done once per node)
    if (base0 <= stall && stall < base0 + kShareRounds * 32) {
      if (has_duplicate(keys, sp.m, lane)) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_DUPLICATE);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        return evals;
      }
    }
    if constexpr (MODE >= 8) {
      if (sp.tail) {
        uint64_t hit;
        evals += shared_block_two_phase<MODE, STAGED>(keys, sp, depth, lane, base0, best, surv, &hit);
        if (hit != ~0ull) {
          if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), hit);
          return evals;
        }
        continue;
      }
    }
    for (uint32_t r = 0; r < kShareRounds; r++) {
      const uint64_t base = base0 + r * 32;
      if (r && base >= volatile_load(best)) return evals;
      const uint64_t kp = family_key(base + lane, depth);
      bool ok = split_trial<MODE, STAGED>(keys, sp, kp);
      if ((MODE == 5 || (MODE >= 7 && sp.confirm)) && ok) ok = split_trial<1, STAGED>(keys, sp, kp);
      const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
      evals += 32 * sp.m;
      if (hits) {
        if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), base + __ffs(hits) - 1);
        return evals;
      }
    }
  }
}

template <bool STAGED>
__device__ __forceinline__ uint64_t shared_search(const uint64_t* __restrict__ keys, const SplitParams& sp, int mode,
                                                  uint32_t depth, uint32_t lane, uint64_t* best, unsigned int* next,
                                                  uint64_t stall, uint64_t limit, int* err, uint4* surv) {
  if (STAGED) {
    switch (mode) {
      case 0: return shared_search_warp<0, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 1: return shared_search_warp<1, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 4: return shared_search_warp<4, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 5: return shared_search_warp<5, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 6: return shared_search_warp<6, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 7: return shared_search_warp<7, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 8: return shared_search_warp<8, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
      case 9: return shared_search_warp<9, true>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
    }
  }
  if (mode == 3) return shared_search_warp<3, STAGED>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
  return shared_search_warp<2, STAGED>(keys, sp, depth, lane, best, next, stall, limit, err, surv);
}

// One CTA per node at a time (all 8 warps): takes nodes of `queue` through
// the work counter, joins open nodes once the queue is empty, and calls
// begin(node) (the whole CTA), search(node, idx) (every warp; claims blocks
// through st.next[idx], lowers st.best[idx]) and, in the last participant to
// leave, close(node, index found).  The node state arrays are sized by the
// queue's capacity.  A node takes at most cap_of(node) CTAs at once.
template <typename Cap, typename Begin, typename Search, typename Close>
__device__ __forceinline__ void shared_nodes(const Node* queue, uint32_t total, const SharedNodes& st,
                                             uint32_t* work_counter, int* error, Cap cap_of, Begin begin,
                                             Search search, Close close) {
  __shared__ uint32_t task, owner, closer, drained;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile uint32_t* vflag = st.flag;
  const uint32_t kNodeOpen = 2 * st.epoch - 1, kNodeClosed = 2 * st.epoch;
  uint32_t joins = 0;  // nodes joined: bounded, so that the kernel ends whatever the timing
  if (threadIdx.x == 0) drained = 0;
  __syncthreads();

  for (;;) {
    if (threadIdx.x == 0) {
      uint32_t idx = total, own = 0;
      if (!*reinterpret_cast<volatile int*>(error) && !drained) {
        const uint32_t i = atomicAdd(work_counter, 1u);
        if (i < total) {
          idx = i;
          own = 1;
          st.best[i] = ~0ull;
          st.next[i] = 0;
          st.refs[i] = 1;
          st.cap[i] = cap_of(queue[i]);
          __threadfence();
          vflag[i] = kNodeOpen;
          reinterpret_cast<volatile uint32_t*>(st.owned)[blockIdx.x] = i + 1;
        } else {
          drained = 1;
        }
      }
      task = idx;
      owner = own;
    }
    __syncthreads();
    if (task >= total && drained && warp == 0 && joins < kMaxJoins && !*reinterpret_cast<volatile int*>(error)) {
      joins++;
      // join the open node with the fewest participants, if any
      for (int attempt = 0; attempt < 8; attempt++) {
        uint32_t pick = total, fewest = ~0u;
        for (uint32_t k0 = 0; k0 < gridDim.x; k0 += 32) {
          const uint32_t k = k0 + lane;
          const uint32_t j = k < gridDim.x ? reinterpret_cast<volatile uint32_t*>(st.owned)[k] - 1 : ~0u;
          uint32_t r = ~0u;
          if (j < total && vflag[j] == kNodeOpen) {
            const uint32_t refs = reinterpret_cast<volatile uint32_t*>(st.refs)[j];
            if (refs < reinterpret_cast<volatile uint32_t*>(st.cap)[j]) r = refs;
          }
          // smallest (refs, node) over the warp
          unsigned long long key = (static_cast<unsigned long long>(r) << 32) | (j < total ? j : 0xFFFFFFFFu);
          for (int o = 16; o; o >>= 1) key = min(key, __shfl_xor_sync(0xFFFFFFFFu, key, o));
          if ((key >> 32) < fewest) {
            fewest = static_cast<uint32_t>(key >> 32);
            pick = static_cast<uint32_t>(key);
          }
        }
        if (fewest == ~0u || pick >= total) break;
        bool ok = false;
        if (lane == 0) {
          atomicAdd(&st.refs[pick], 1u);
          __threadfence();
          ok = vflag[pick] == kNodeOpen;
          if (!ok) atomicSub(&st.refs[pick], 1u);  // closed meanwhile
        }
        if (__shfl_sync(0xFFFFFFFFu, ok, 0)) {
          if (lane == 0) task = pick;
          break;
        }
      }
    }
    __syncthreads();
    const uint32_t idx = task;
    if (idx >= total) break;
    const Node nd = queue[idx];
    begin(nd);
    __syncthreads();
    search(nd, idx);
    __syncthreads();
    if (threadIdx.x == 0) {
      // leave; the last participant closes the node
      __threadfence();
      const uint32_t left = atomicSub(&st.refs[idx], 1u);
      closer = left == 1 && atomicCAS(&st.flag[idx], kNodeOpen, kNodeClosed) == kNodeOpen;
      if (owner) reinterpret_cast<volatile uint32_t*>(st.owned)[blockIdx.x] = 0;
    }
    __syncthreads();
    if (closer) {
      const uint64_t found = volatile_load(&st.best[idx]);
      if (found == ~0ull) {
        if (threadIdx.x == 0) set_error(error, RECSPLIT_E_SEARCH_LIMIT);
      } else if (!*reinterpret_cast<volatile int*>(error)) {
        close(nd, found);
      }
    }
    __syncthreads();
  }
}

// Participants worth having on a split node: one CTA per 2^10 expected trials
// (a CTA's warps test 1024 indices at a time), at most 16: what more of them
// test lies beyond the index found and takes issue slots from other nodes (16
// on nodes of 3679 trials, l = 12, b = 2000: split phase 2.8 -> 4.7 ms).
template <bool COUNT>
__global__ void __launch_bounds__(kThreads, 4) k_split_shared(SearchArgs a, SharedNodes st, uint32_t cap,
                                                              uint32_t tables) {
  extern __shared__ __align__(16) uint64_t dynamic[];  // tables of modes 8 and 9 if any, then the node's keys
  __shared__ uint32_t fill[16];
  __shared__ uint4 surv[kWarps][kShareRounds * 32];  // two-phase block survivors, per warp
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long evals = 0;  // work counting: evaluations of this warp, flushed at exit
  const uint32_t* const counts = tables ? reinterpret_cast<const uint32_t*>(dynamic) : nullptr;
  if (tables) fill_part_counts(reinterpret_cast<uint32_t*>(dynamic));
  uint64_t* const mine = dynamic + (tables ? kPartCounts : 0);
  shared_nodes(
      a.split_in[1], *a.split_in_count[1], st, a.work_counter, a.error,
      [&](const Node& nd) {
        const uint64_t et = a.table[nd.depth >> 8][kTableWords * nd.m + 2];
        return static_cast<uint32_t>(min(uint64_t(16), max(uint64_t(1), et >> 10)));
      },
      [&](const Node& nd) {
        const uint64_t* src = a.keys[nd.depth & 1] + nd.start;
        if (nd.m <= cap)
          for (uint32_t j = threadIdx.x; j < nd.m; j += kThreads) mine[j] = src[j];
        if (threadIdx.x < 16) fill[threadIdx.x] = 0;
      },
      [&](const Node& nd, uint32_t idx) {
        const uint32_t depth = nd.depth & kDepthMask;
        const uint64_t* table = a.table[nd.depth >> 8];
        SplitParams sp;
        const int mode = split_setup(nd, table, counts, sp);
        const uint64_t stall = stall_threshold(table, nd.m), limit = trial_limit(table, nd.m);
        const uint64_t done =
            nd.m <= cap ? shared_search<true>(mine, sp, mode, depth, lane, &st.best[idx], &st.next[idx], stall, limit,
                                              a.error, surv[warp])
                        : shared_search<false>(a.keys[depth & 1] + nd.start, sp, mode, depth, lane, &st.best[idx],
                                               &st.next[idx], stall, limit, a.error, surv[warp]);
        if (COUNT) evals += done;
      },
      [&](const Node& nd, uint64_t seed) {
        partition_node(a, nd, seed, nd.m <= cap ? mine : nullptr, threadIdx.x, kThreads, lane, warp == 0, fill);
      });
  if (COUNT && lane == 0 && evals) atomicAdd(a.exec_count + 1, evals);
}

// ---------------------------------------------------------------- leaves
// Leaf of exactly L keys (the common case): keys in registers, bijection
// test as a sum of one-hot bits compared with 2^L - 1.  A sum of k powers of
// two has k one bits only if no two of them are equal (every carry merges
// two one bits), and 2^L - 1 has L one bits, so the sum of the L one-hot
// values equals 2^L - 1 exactly when the values are distinct.  The sum, unlike
// an OR, can be issued to the multiply-add pipe as well as the integer ALU.
template <int L>
__device__ __forceinline__ bool leaf_trial_full(const uint64_t (&x)[L], uint64_t kp) {
  uint32_t seen = 0;
#pragma unroll
  for (int j = 0; j < L; j++) seen += 1u << phi_fixed<L>(x[j], kp);
  return seen == (L == 32 ? ~0u : ((1u << L) - 1));
}

// The family key of index i at depth d, (i * 64 + d) * W, is i * 64W + d W:
// a lane's keys for indices 32 apart differ by 32 * 64W, one 64-bit add.
constexpr uint64_t kWeyl64 = kWeyl << 6;
constexpr uint64_t kLaneStep = kWeyl64 * 32;

__device__ __forceinline__ uint64_t index_key(uint64_t index, uint64_t dkey) { return index * kWeyl64 + dkey; }

// Two-phase round of a warp over the indices base + j * 32 + lane, j < spl,
// for a leaf of exactly L keys.  Phase 1 maps the first H keys: an index whose
// first H values are not distinct cannot be a bijection.  The survivors are
// compacted, in index order, into the warp's shared buffer with their
// partial one-hot sums (H one bits) and their pre-shifted keys; phase 2
// finishes them on the last L - H keys, 32 at a time.  The first survivor
// that completes 2^L - 1 is the smallest bijective index of the round.
// Returns it, or ~0 if the round has none.  With `exec` set, the
// evaluations the round executed are added to it (work counting).
//
// H minimises the expected work per index, H + P_H (L - H) evaluations plus
// the compaction and reload of a survivor (costed as 2.5 evaluations), with
// P_H = L! / ((L - H)! L^H) the probability that the first H values are
// distinct: 5 of 8 keys, 7 of 12, 8 of 16, 10 of 24.
__host__ __device__ constexpr int leaf_first_part(int l) {
  double p = 1.0, best = 1e30;
  int arg = 1;
  for (int h = 1; h < l; h++) {
    const double cost = h + p * (l - h) + 2.5 * p;
    if (cost < best) {
      best = cost;
      arg = h;
    }
    p = p * (l - h) / l;
  }
  return arg;
}
constexpr uint32_t kMaxSpl = 8;

template <int L>
__device__ __forceinline__ uint64_t leaf_round_two_phase(const uint64_t (&x)[L], uint64_t base, uint64_t dkey,
                                                         uint32_t spl, uint32_t lane, uint4* surv,
                                                         unsigned long long* exec) {
  constexpr int H = leaf_first_part(L);
  constexpr uint32_t full = L == 32 ? ~0u : ((1u << L) - 1);
  const uint32_t below = (1u << lane) - 1;
  uint32_t nsurv = 0;
  uint64_t k = index_key(base + lane, dkey);
#pragma unroll 4
  for (uint32_t j = 0; j < spl; j++, k += kLaneStep) {
    const uint64_t kp = k ^ (k >> 30);
    uint32_t seen = 0;
#pragma unroll
    for (int i = 0; i < H; i++) seen += 1u << phi_fixed<L>(x[i], kp);
    const bool ok = __popc(seen) == H;
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, ok);
    if (ok)
      surv[nsurv + __popc(b & below)] =
          make_uint4(j * 32 + lane, seen, static_cast<uint32_t>(kp), static_cast<uint32_t>(kp >> 32));
    nsurv += __popc(b);
  }
  __syncwarp();
  uint64_t win = ~0ull;
  uint32_t done = 0;
  for (uint32_t t0 = 0; t0 < nsurv; t0 += 32) {
    const uint32_t t = t0 + lane;
    bool ok = false;
    if (t < nsurv) {
      const uint4 e = surv[t];
      const uint64_t kp = (uint64_t(e.w) << 32) | e.z;
      uint32_t seen = e.y;
#pragma unroll
      for (int i = H; i < L; i++) seen += 1u << phi_fixed<L>(x[i], kp);
      ok = seen == full;
    }
    done = min(nsurv, t0 + 32);
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, ok);
    if (b) {
      win = base + surv[t0 + __ffs(b) - 1].x;
      break;
    }
  }
  if (exec && lane == 0) *exec += spl * 32 * H + done * (L - H);
  __syncwarp();
  return win;
}

// Three-phase test for full leaves of L >= kFifoLeaf keys, with the
// survivors of each phase kept, in index order, in first-in first-out
// buffers of the warp that outlive the round: phase 1 maps the first h1 keys
// of the round's spl * 32 indices and appends the survivors to A; phase 2
// maps keys h1 .. h2 - 1 of 32 entries of A at a time and appends its
// survivors to B; phase 3 finishes 32 entries of B at a time.  A batch runs
// only once its buffer holds 32 entries, so every phase works on full
// warps (the two-phase round above finishes its few survivors, about 0.12 of
// 32 * spl at l = 16, in a mostly idle batch every round).  Entries leave
// each buffer in the order they entered it and every entry of B is older
// than every entry of A, so the first index that phase 3 completes is the
// smallest bijective index among all the indices the warp has generated.
// When the warp stops (another warp of its group found a smaller index, or
// the trial limit) it first drains both buffers with partial batches.
//
// h1 < h2 minimise the expected work per index, h1 + P_h1 (h2 - h1 + c) +
// P_h2 (l - h2 + c) evaluations with c = 2.5 for the compaction and reload of
// a survivor (P_h as above): (6, 9) at l = 13, (8, 13) at 24.
// At l = 12 a leaf takes about 2 * 10^4 trials, a few rounds of a group, and
// draining the buffers at the end of every leaf costs more than the full
// batches save (measured: 6% slower than the two-phase round), so the
// buffers start at 13 keys.
struct LeafPhases {
  int h1, h2;
};
__host__ __device__ constexpr LeafPhases leaf_phases(int l) {
  if (l == 16) return LeafPhases{6, 9};  // whole triples (below), 1% above the minimum
  double best = 1e30;
  LeafPhases arg{1, 2};
  double p1 = 1.0;  // P_h1
  for (int h1 = 1; h1 < l - 1; h1++) {
    double p2 = p1;  // P_h2
    for (int h2 = h1 + 1; h2 < l; h2++) {
      p2 = p2 * (l - (h2 - 1)) / l;
      const double cost = h1 + p1 * (h2 - h1 + 2.5) + p2 * (l - h2 + 2.5);
      if (cost < best) {
        best = cost;
        arg = LeafPhases{h1, h2};
      }
    }
    p1 = p1 * (l - h1) / l;
  }
  return arg;
}
constexpr int kFifoLeaf = 13;
constexpr uint32_t kFifoA = 32 * kMaxSpl + 32;  // below 32 left + one round's spl * 32
constexpr uint32_t kFifoB = 64;                 // below 32 left + one batch of A
//
// At l = 16 the values of three keys, 4 bits each, are shifted into one word
// (one funnel shift per key instead of two shifts and an add), and a table in
// shared memory gives the set of the three, or all ones when two are equal;
// sets are combined by testing that they share no value.
//
// An entry is {low 32 bits of the index, set of the values so far}; the
// function key is computed again from the index, 8 instructions per entry of a
// full batch, which costs no more than storing and loading it did and halves
// the buffers.

// Set of the values of a 12-bit index (three 4-bit values), 0xFFFF when two are
// equal: two consecutive entries per 32-bit word.
__device__ __forceinline__ void fill_hex_sets(uint32_t* lut) {
  for (uint32_t w = threadIdx.x; w < 2048; w += kThreads) {
    const uint32_t e = w * 2;
    const uint32_t p = (1u << (e >> 8)) | (1u << ((e >> 4) & 15));
    const bool distinct = __popc(p) == 2;
    uint32_t v = 0;
#pragma unroll
    for (uint32_t t = 0; t < 2; t++) {
      const uint32_t bit = 1u << ((e + t) & 15);
      v |= (distinct && !(p & bit) ? p | bit : 0xFFFFu) << (16 * t);
    }
    lut[w] = v;
  }
}

// l = 16: the set of the values of keys x[I], x[I + 1], x[I + 2].
template <int I>
__device__ __forceinline__ uint32_t hex_set(const uint64_t* x, uint64_t kp, const uint16_t* lut) {
  uint32_t v = family_top32(x[I], kp) >> 28;
  v = __funnelshift_l(family_top32(x[I + 1], kp), v, 4);
  v = __funnelshift_l(family_top32(x[I + 2], kp), v, 4);
  return lut[v];
}

// The keys of the leaf are read from shared memory: 2 l registers for them
// held the kernel to three CTAs per SM, too few for its dependent chains (ncu
// at l = 16, 24 warps per SM: issue 66%, fixed-latency waits the leading
// stall).  Leaf phase at l = 16, b = 2000, 4 * 10^5 keys, four warps per leaf:
// 143 ms with 16-byte entries and keys in registers, 131 ms so with four CTAs
// per SM, 139 ms with five (48 registers), 155 ms with six.

// Moves entries [r, n) of a warp buffer, fewer than 32, to its front.
__device__ __forceinline__ uint32_t fifo_compact(uint2* buf, uint32_t r, uint32_t n, uint32_t lane) {
  const uint32_t rem = n - r;
  uint2 v = make_uint2(0, 0);
  if (lane < rem) v = buf[r + lane];
  __syncwarp();
  if (lane < rem) buf[lane] = v;
  __syncwarp();
  return rem;
}

// Index of an entry from its low 32 bits and the newest index generated.
__device__ __forceinline__ uint64_t fifo_index(uint32_t low, uint64_t newest) {
  return newest - static_cast<uint32_t>(static_cast<uint32_t>(newest) - low);
}

__device__ __forceinline__ uint64_t fifo_key(uint32_t low, uint64_t newest, uint64_t dkey) {
  const uint64_t k = index_key(fifo_index(low, newest), dkey);
  return k ^ (k >> 30);
}

template <int L>
__device__ __forceinline__ void fifo_phase1(const uint64_t* x, uint64_t base, uint64_t dkey, uint32_t spl,
                                            uint32_t lane, const uint16_t* lut, uint2* a, uint32_t& na) {
  constexpr int H1 = leaf_phases(L).h1;
  const uint32_t below = (1u << lane) - 1;
  uint64_t k = index_key(base + lane, dkey);
  for (uint32_t j = 0; j < spl; j++, k += kLaneStep) {
    const uint64_t kp = k ^ (k >> 30);
    uint32_t seen = 0;
    bool ok;
    if constexpr (L == 16) {
      const uint32_t s0 = hex_set<0>(x, kp, lut), s1 = hex_set<3>(x, kp, lut);
      ok = !(s0 & s1);
      seen = s0 | s1;
    } else {
#pragma unroll
      for (int i = 0; i < H1; i++) seen += 1u << phi_fixed<L>(x[i], kp);
      ok = __popc(seen) == H1;
    }
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, ok);
    if (ok) a[na + __popc(b & below)] = make_uint2(static_cast<uint32_t>(base) + j * 32 + lane, seen);
    na += __popc(b);
  }
  __syncwarp();
}

// Phase 2 on entries [ra, ra + c) of A (c <= 32); survivors go to B.
template <int L>
__device__ __forceinline__ void fifo_phase2(const uint64_t* x, const uint2* a, uint32_t ra, uint32_t c,
                                            uint64_t newest, uint64_t dkey, uint32_t lane, const uint16_t* lut,
                                            uint2* b, uint32_t& nb) {
  constexpr LeafPhases ph = leaf_phases(L);
  uint2 e = make_uint2(0, 0);
  bool ok = false;
  if (lane < c) {
    e = a[ra + lane];
    const uint64_t kp = fifo_key(e.x, newest, dkey);
    if constexpr (L == 16) {
      const uint32_t s = hex_set<6>(x, kp, lut);
      ok = !(e.y & s);
      e.y |= s;
    } else {
#pragma unroll
      for (int i = ph.h1; i < ph.h2; i++) e.y += 1u << phi_fixed<L>(x[i], kp);
      ok = __popc(e.y) == ph.h2;
    }
  }
  const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
  if (ok) b[nb + __popc(hits & ((1u << lane) - 1))] = e;
  nb += __popc(hits);
  __syncwarp();
}

// Phase 3 on entries [rb, rb + c) of B; on success `low` is the low 32 bits
// of the first bijective entry's index.
template <int L>
__device__ __forceinline__ bool fifo_phase3(const uint64_t* x, const uint2* b, uint32_t rb, uint32_t c,
                                            uint64_t newest, uint64_t dkey, uint32_t lane, const uint16_t* lut,
                                            uint32_t& low) {
  constexpr int H2 = leaf_phases(L).h2;
  constexpr uint32_t full = L == 32 ? ~0u : ((1u << L) - 1);
  bool ok = false;
  uint32_t id = 0;
  if (lane < c) {
    const uint2 e = b[rb + lane];
    const uint64_t kp = fifo_key(e.x, newest, dkey);
    uint32_t seen = e.y;
    if constexpr (L == 16) {
      const uint32_t s0 = hex_set<9>(x, kp, lut), s1 = hex_set<12>(x, kp, lut);
      ok = !(seen & s0);
      seen |= s0;
      ok = ok && !(seen & s1);
      seen |= s1;
      ok = ok && !(seen & (1u << phi_fixed<L>(x[15], kp)));
    } else {
#pragma unroll
      for (int i = H2; i < L; i++) seen += 1u << phi_fixed<L>(x[i], kp);
      ok = seen == full;
    }
    id = e.x;
  }
  const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
  if (!hits) return false;
  low = __shfl_sync(0xFFFFFFFFu, id, __ffs(hits) - 1);
  return true;
}

// Phases 2 and 3 on the full batches of the warp's buffers (on every entry
// with `drain`).  `newest` is the largest index generated so far.  Returns
// the smallest bijective index found, or ~0.
template <int L>
__device__ __forceinline__ uint64_t fifo_pump(const uint64_t* x, uint2* a, uint32_t& na, uint2* b, uint32_t& nb,
                                              bool drain, uint64_t newest, uint64_t dkey, uint32_t lane,
                                              const uint16_t* lut, unsigned long long* exec) {
  constexpr LeafPhases ph = leaf_phases(L);
  uint32_t ra = 0, low = 0;
  bool found = false;
  while (!found && (na - ra >= 32 || (drain && na > ra))) {
    const uint32_t c = min(32u, na - ra);
    fifo_phase2<L>(x, a, ra, c, newest, dkey, lane, lut, b, nb);
    if (exec && lane == 0) *exec += c * (ph.h2 - ph.h1);
    ra += c;
    uint32_t rb = 0;
    while (nb - rb >= 32) {
      if (exec && lane == 0) *exec += 32 * (L - ph.h2);
      if ((found = fifo_phase3<L>(x, b, rb, 32, newest, dkey, lane, lut, low))) break;
      rb += 32;
    }
    if (!found && rb) nb = fifo_compact(b, rb, nb, lane);
  }
  if (!found) {
    if (ra) na = fifo_compact(a, ra, na, lane);  // fewer than 32 left unless draining, which leaves none
    for (uint32_t rb = 0; drain && rb < nb; rb += 32) {
      const uint32_t c = min(32u, nb - rb);
      if (exec && lane == 0) *exec += c * (L - ph.h2);
      if ((found = fifo_phase3<L>(x, b, rb, c, newest, dkey, lane, lut, low))) break;
    }
    if (drain) nb = 0;
  }
  if (!found) return ~0ull;
  return fifo_index(low, newest);
}

// Blocks per SM the register budget must allow (keys live in registers).
__host__ __device__ constexpr int leaf_min_blocks(int l) { return l <= 5 ? 5 : (l <= 12 ? 4 : 3); }

// Leaf of M keys of the perfect, non-minimal variant: the values in [0, range),
// range = M + extra, must be distinct, i.e. the sum of the one-hot values
// must have M one bits (a sum of powers of two loses one bits on every
// carry, and a carry out of bit 31 only lowers the count further).
template <int M>
__device__ __forceinline__ bool leaf_trial_range(const uint64_t (&x)[M], uint32_t range, uint64_t kp) {
  uint32_t seen = 0;
#pragma unroll
  for (int j = 0; j < M; j++) seen += 1u << phi_pre(x[j], kp, range);
  return __popc(seen) == M;
}

// Search of one leaf of M keys by a group of gwarps warps (this is warp wig):
// lowers *best (shared memory, ~0 on entry) to the first successful index.
enum LeafTest { kOnePhase, kTwoPhases, kRangeTest };

template <int M, LeafTest TEST>
__device__ __forceinline__ void search_leaf(const uint64_t* __restrict__ src, uint32_t depth,
                                            const uint64_t* table, uint32_t range, uint32_t spl, uint32_t wig,
                                            uint32_t gwarps, uint32_t lane, uint64_t* best, uint4* surv, int* err,
                                            unsigned long long* exec) {
  uint64_t x[M];
#pragma unroll
  for (int j = 0; j < M; j++) x[j] = __ldg(src + j);
  const uint64_t stall = stall_threshold(table, M);
  const uint64_t limit = trial_limit(table, M);
  const uint64_t dkey = uint64_t(depth) * kWeyl;
  uint32_t rounds = 0;
  // a round of a warp covers the spl * 32 indices from base; lane L tests
  // base + j * 32 + L for j < spl
  const uint64_t span = uint64_t(spl) * 32;
  // one compare per round: the stall point until it is checked, then the limit
  for (uint64_t base = uint64_t(wig) * span, next_check = min(stall, limit);; base += uint64_t(gwarps) * span) {
    if (gwarps > 1 && __any_sync(0xFFFFFFFFu, base >= volatile_load(best))) break;
    if ((++rounds & 255) == 0 && __shfl_sync(0xFFFFFFFFu, lane == 0 ? *reinterpret_cast<volatile int*>(err) : 0, 0))
      break;  // another search failed, or the host cancelled the build
    if (base >= next_check) {
      if (base >= limit) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_SEARCH_LIMIT);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        break;
      }
      next_check = limit;
      bool dup = false;
#pragma unroll
      for (int i = 0; i < M; i++)
#pragma unroll
        for (int j = i + 1; j < M; j++) dup |= x[i] == x[j];
      if (dup) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_DUPLICATE);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        break;
      }
    }
    uint64_t found = ~0ull;
    if constexpr (TEST == kTwoPhases) {
      found = leaf_round_two_phase<M>(x, base, dkey, spl, lane, surv, exec);
    } else {
      uint64_t k = index_key(base + lane, dkey);
      for (uint32_t j = 0; j < spl; j++, k += kLaneStep) {
        const uint64_t kp = k ^ (k >> 30);
        const bool ok = TEST == kRangeTest ? leaf_trial_range<M>(x, range, kp) : leaf_trial_full<M>(x, kp);
        const uint32_t hits = __ballot_sync(0xFFFFFFFFu, ok);
        if (hits && found == ~0ull) found = base + j * 32 + __ffs(hits) - 1;
      }
      if (exec && lane == 0) *exec += spl * 32 * M;
    }
    if (found != ~0ull) {
      if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), found);
      break;
    }
  }
}

// Leaf of m keys, 2 <= m <= LMAX, by the search for exactly m keys (a search
// over LMAX masked slots evaluates LMAX keys whatever m is: the partial leaves
// of 2 to 11 keys at l = 12 took 1.87 ms of a batched build so, in 16 slots).
// From 6 keys on the two-phase test, with the indices per lane that its trial
// count calls for.
template <int M, int LMAX, bool RANGE>
__device__ __forceinline__ void search_leaf_of(uint32_t m, const uint64_t* __restrict__ src, uint32_t depth,
                                               const uint64_t* table, uint32_t range, uint32_t wig, uint32_t gwarps,
                                               uint32_t lane, uint64_t* best, uint4* surv, int* err,
                                               unsigned long long* exec) {
  if (m == M) {
    constexpr LeafTest test = RANGE ? kRangeTest : (M >= 6 ? kTwoPhases : kOnePhase);
    constexpr uint32_t spl = RANGE || M < 6 ? 1 : (M == 6 ? 2 : (M < 9 ? 4 : 8));
    search_leaf<M, test>(src, depth, table, range, spl, wig, gwarps, lane, best, surv, err, exec);
  } else if constexpr (M < LMAX) {
    search_leaf_of<M + 1, LMAX, RANGE>(m, src, depth, table, range, wig, gwarps, lane, best, surv, err, exec);
  }
}

// Full leaves of L keys (PART false), or leaves of 2 to L keys of the class's
// full (qfull) or partial queue.  RANGE: perfect, non-minimal variant (leaf
// range m + extra of the class).
template <int L, bool PART, bool TWO, bool RANGE = false>
__global__ void __launch_bounds__(kThreads, leaf_min_blocks(L)) k_leaves(SearchArgs a, uint32_t gwarps,
                                                                         uint32_t chunk, uint32_t spl,
                                                                         uint32_t qfull) {
  __shared__ uint64_t best[kWarps];
  __shared__ uint32_t task[kWarps];
  __shared__ unsigned long long wexec[kWarps];  // work counting: evaluations per warp, flushed at exit
  constexpr bool kSurvivors = PART ? !RANGE && L >= 6 : TWO && L >= 4;
  __shared__ uint4 surv[kSurvivors ? kWarps : 1][kSurvivors ? 32 * kMaxSpl : 1];  // one round's survivors
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long* const exec = a.exec_count ? &wexec[warp] : nullptr;
  if (lane == 0) wexec[warp] = 0;
  const Node* queue = !PART || qfull ? a.full_q[a.cls] : a.part_q[a.cls];
  const uint32_t total = !PART || qfull ? a.full_n[a.cls] : a.part_n[a.cls];
  gwarps = group_warps(gwarps, total, PART ? 2 : group_spread(a.table[a.cls][kTableWords * L + 2]));
  const uint32_t groups = gridDim.x * (kWarps / gwarps);
  chunk = min(chunk, max(1u, total / (2 * groups)));
  const uint32_t gid = warp / gwarps, wig = warp % gwarps;
  const bool leader = wig == 0 && lane == 0;
  const uint32_t extra = RANGE ? a.extra_of[a.cls] : 0;
  const uint64_t* table = a.table[a.cls];
  uint4* const mine = surv[kSurvivors ? warp : 0];

  for (;;) {
    if (leader) task[gid] = *reinterpret_cast<volatile int*>(a.error) ? total : atomicAdd(a.work_counter, chunk);
    group_sync(gid, gwarps);
    const uint32_t first = task[gid];
    if (first >= total) break;
    const uint32_t last = min(total, first + chunk);
    for (uint32_t idx = first; idx < last; idx++) {
      const Node nd = queue[idx];
      const uint32_t depth = nd.depth & kDepthMask;
      const uint64_t* src = a.keys[depth & 1] + nd.start;
      if (leader) best[gid] = ~0ull;
      group_sync(gid, gwarps);
      if constexpr (PART)
        search_leaf_of<2, L, RANGE>(nd.m, src, depth, table, nd.m + extra, wig, gwarps, lane, &best[gid], mine,
                                    a.error, exec);
      else
        search_leaf<L, TWO && L >= 4 ? kTwoPhases : kOnePhase>(src, depth, table, L, spl, wig, gwarps, lane,
                                                               &best[gid], mine, a.error, exec);
      group_sync(gid, gwarps);
      if (leader) {
        a.seeds[nd.slot] = best[gid];
        a.sizes[nd.slot] = nd.m;
      }
      group_sync(gid, gwarps);
    }
  }
  if (exec && lane == 0 && wexec[warp]) atomicAdd(a.exec_count, wexec[warp]);
}

// ---------------------------------------------------------------- shared leaves
// Full leaves of kFifoLeaf keys or more with the three-phase test, one CTA per
// leaf; a CTA that finds the queue empty joins a leaf in progress, as for
// shared split nodes.  Trial counts are geometric (873,000 on average at
// l = 16): with four warps per leaf and no joining, 62,700 leaves kept a tenth
// of the warps idle on average, and 6,000 leaves a third.  Every warp claims
// kLeafShareRounds rounds of indices at a time, in increasing order, so its
// buffers stay in index order and every index below the final best has been
// tested.
constexpr uint32_t kLeafShareRounds = 4;

// One warp's part in the search of one leaf.
template <int L>
__device__ __forceinline__ void fifo_search(const uint64_t* x, uint32_t depth, uint32_t spl, uint64_t stall,
                                            uint64_t limit, uint64_t* best, unsigned int* next, int* err,
                                            uint32_t lane, const uint16_t* lut, uint2* fa, uint2* fb,
                                            unsigned long long* exec) {
  const uint64_t dkey = uint64_t(depth) * kWeyl;
  const uint64_t span = uint64_t(spl) * 32, block = kLeafShareRounds * span;
  uint64_t base = 0, end = 0, newest = 0, mark = 0;
  uint32_t na = 0, nb = 0, rounds = 0;
  for (;;) {
    bool drain = false, generate = true;
    if (base == end) {
      unsigned int blk = 0;
      if (lane == 0) blk = atomicAdd(next, 1u);
      base = uint64_t(__shfl_sync(0xFFFFFFFFu, blk, 0)) * block;
      end = base + block;
      // the one warp whose block holds the stall point checks for keys that
      // can never be separated
      if (base <= stall && stall < end && has_duplicate(x, L, lane)) {
        if (lane == 0) {
          set_error(err, RECSPLIT_E_DUPLICATE);
          atomicMin(reinterpret_cast<unsigned long long*>(best), 0ull);
        }
        return;
      }
      // an entry holds the low 32 bits of its index: none may stay until the
      // newest index is 2^32 beyond it
      if (end - mark >= (1ull << 32)) {
        drain = true;
        generate = false;
        mark = base;
      }
    }
    // a smaller index is known, or the limit is reached (the closer reports it
    // if no index below it succeeded): finish what waits in the buffers
    const bool last = __any_sync(0xFFFFFFFFu, base >= volatile_load(best)) || base >= limit;
    if (last) {
      drain = true;
      generate = false;
    }
    if ((++rounds & 255) == 0 && __shfl_sync(0xFFFFFFFFu, lane == 0 ? *reinterpret_cast<volatile int*>(err) : 0, 0))
      return;  // another search failed, or the host cancelled the build
    if (generate) {
      fifo_phase1<L>(x, base, dkey, spl, lane, lut, fa, na);
      if (exec && lane == 0) *exec += span * leaf_phases(L).h1;
      base += span;
      newest = base - 1;
    }
    const uint64_t found = na || nb ? fifo_pump<L>(x, fa, na, fb, nb, drain, newest, dkey, lane, lut, exec) : ~0ull;
    if (found != ~0ull) {
      if (lane == 0) atomicMin(reinterpret_cast<unsigned long long*>(best), found);
      return;
    }
    if (last) return;
  }
}

template <int L>
__global__ void __launch_bounds__(kThreads, 4) k_leaves_shared(SearchArgs a, SharedNodes st, uint32_t spl) {
  __shared__ uint64_t x[L];
  __shared__ uint2 fifo[kWarps][kFifoA + kFifoB];
  __shared__ uint32_t lut[L == 16 ? 2048 : 1];
  __shared__ unsigned long long wexec[kWarps];  // work counting: evaluations per warp, flushed at exit
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) wexec[warp] = 0;
  if (L == 16) fill_hex_sets(lut);
  const uint64_t* table = a.table[a.cls];
  const uint64_t stall = stall_threshold(table, L), limit = trial_limit(table, L);
  // participants worth having: one CTA per 2^12 expected trials, at most 16
  const uint32_t cap = static_cast<uint32_t>(min(uint64_t(16), max(uint64_t(1), table[kTableWords * L + 2] >> 12)));
  shared_nodes(
      a.full_q[a.cls], a.full_n[a.cls], st, a.work_counter, a.error, [&](const Node&) { return cap; },
      [&](const Node& nd) {
        if (threadIdx.x < L) x[threadIdx.x] = a.keys[nd.depth & 1][nd.start + threadIdx.x];
      },
      [&](const Node& nd, uint32_t idx) {
        fifo_search<L>(x, nd.depth & kDepthMask, spl, stall, limit, &st.best[idx], &st.next[idx], a.error, lane,
                       reinterpret_cast<const uint16_t*>(lut), fifo[warp], fifo[warp] + kFifoA,
                       a.exec_count ? &wexec[warp] : nullptr);
      },
      [&](const Node& nd, uint64_t found) {
        if (threadIdx.x == 0) {
          a.seeds[nd.slot] = found;
          a.sizes[nd.slot] = L;
        }
      });
  if (a.exec_count && lane == 0 && wexec[warp]) atomicAdd(a.exec_count, wexec[warp]);
}

// ---------------------------------------------------------------- packed leaves
// Full leaves of 4 to 8 keys.  A leaf of 8 keys takes 416 trials on
// average, so a warp that tests 128 indices of one leaf per round tests 64
// beyond the winner (15%).  Here a warp holds up to four leaves, eight lanes
// on each: a round tests 8 spl indices per leaf, and the survivors of the
// first H keys of all four are finished together, 32 at a time, so the second
// phase's batches stay as full as with one leaf.  A leaf that finishes is
// replaced at once from nodes the warp has taken ahead (one atomic and one
// load per chunk).  At the end of the queue, and when there are too few
// leaves for all warps, the lanes of free slots join the leaves that remain.
//
// The keys of the lane's leaf are in its registers, copies in shared memory
// serve the second phase.  A round covers every index of [base, base +
// lanes * spl) of its leaf and all survivors are finished, so the smallest
// success of the round is the leaf's first bijective index.
//
// At 8 keys the first four values, 3 bits each, are shifted into one word
// (one funnel shift per key instead of two shifts and an add) and a table of
// 4096 bytes in shared memory gives the set of the four values, or 0xFF when
// two are equal.
constexpr int kPackedLeaf = 8;
constexpr uint32_t kPackedSlots = 4;

// Set of the values of a 12-bit index (four 3-bit values), 0xFF when two are
// equal: four consecutive entries (the index's low 2 bits) per 32-bit word.
__device__ __forceinline__ void fill_octal_sets(uint32_t* lut) {
  for (uint32_t w = threadIdx.x; w < 1024; w += kThreads) {
    const uint32_t e = w * 4;
    const uint32_t p = (1u << (e >> 9)) | (1u << ((e >> 6) & 7)) | (1u << ((e >> 3) & 7));
    const bool distinct = __popc(p) == 3;
    uint32_t v = 0;
#pragma unroll
    for (uint32_t t = 0; t < 4; t++) {
      const uint32_t bit = 1u << ((e + t) & 7);
      v |= (distinct && !(p & bit) ? p | bit : 0xFFu) << (8 * t);
    }
    lut[w] = v;
  }
}

// Whether the first H values of index key kp are distinct, and their set.
template <int L, int H>
__device__ __forceinline__ bool leaf_head(const uint64_t (&x)[L], uint64_t kp, const uint8_t* lut, uint32_t& seen) {
  if constexpr (L == 8 && H >= 4) {
    uint32_t v = family_top32(x[0], kp) >> 29;
#pragma unroll
    for (int i = 1; i < 4; i++) v = __funnelshift_l(family_top32(x[i], kp), v, 3);
    seen = lut[v];
    bool ok = H > 4 || seen != 0xFFu;
#pragma unroll
    for (int i = 4; i < H; i++) {
      const uint32_t bit = 1u << phi_fixed<L>(x[i], kp);
      ok = ok && !(seen & bit);
      seen |= bit;
    }
    return ok;
  } else {
    seen = 0;
#pragma unroll
    for (int i = 0; i < H; i++) seen += 1u << phi_fixed<L>(x[i], kp);
    return __popc(seen) == H;
  }
}

// RANGE: perfect, non-minimal variant (range L + extra of the class).  Its
// leaves, and bijections of at most 5 keys, take a few dozen trials: one phase.
template <int L, bool RANGE>
__global__ void __launch_bounds__(kThreads, 4) k_leaves_packed(SearchArgs a, uint32_t chunk, uint32_t spl) {
  constexpr bool kOne = RANGE || L <= 5;
  constexpr int H = kOne ? L : leaf_first_part(L);
  constexpr bool kLut = L == 8 && !RANGE;
  constexpr uint32_t full = (1u << L) - 1;
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  __shared__ uint64_t skeys[kWarps][kPackedSlots][L];
  __shared__ uint64_t sdkey[kWarps][kPackedSlots];
  __shared__ uint32_t sbase[kWarps][kPackedSlots], sbest[kWarps][kPackedSlots];
  __shared__ uint2 surv[kOne ? 1 : kWarps][kOne ? 1 : 32 * kMaxSpl];  // {index, set of the first values | slot << 16}
  __shared__ uint32_t lut[kLut ? 1024 : 1];
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t total = a.full_n[a.cls];
  if (kLut) fill_octal_sets(lut);
  __syncthreads();
  const Node* queue = a.full_q[a.cls];
  const uint32_t range = L + (RANGE ? a.extra_of[a.cls] : 0);
  const uint32_t below = (1u << lane) - 1;
  const uint32_t nwarps = gridDim.x * kWarps;
  const uint32_t slots = total >= kPackedSlots * nwarps ? kPackedSlots : (total >= 2 * nwarps ? 2 : 1);
  chunk = min(min(chunk, 32u), max(1u, total / (4 * nwarps)));
  const uint32_t stall = static_cast<uint32_t>(min(stall_threshold(a.table[a.cls], L), uint64_t(1) << 31));
  const uint32_t limit = static_cast<uint32_t>(min(trial_limit(a.table[a.cls], L), uint64_t(1) << 31));

  Node pend{};                    // lane i: node i of the chunk taken
  uint32_t pend_at = 0, pend_n = 0;
  bool more = true;
  uint32_t act = 0;               // slots in use
  uint32_t my_slot = 0;           // lanes 0..3: code slot of the leaf in slot `lane`
  uint32_t rounds = 0;
  unsigned long long exec = 0;

  for (;;) {
    // fill free slots
    for (uint32_t need = ~act & ((1u << slots) - 1); need && more; need &= need - 1) {
      if (pend_at == pend_n) {
        uint32_t first = 0;
        if (lane == 0) first = *reinterpret_cast<volatile int*>(a.error) ? total : atomicAdd(a.work_counter, chunk);
        first = __shfl_sync(kAll, first, 0);
        if (first >= total) {
          more = false;
          break;
        }
        pend_n = min(chunk, total - first);
        pend_at = 0;
        if (lane < pend_n) pend = queue[first + lane];
      }
      const uint32_t q = __ffs(need) - 1;
      const uint32_t start = __shfl_sync(kAll, pend.start, pend_at), slot = __shfl_sync(kAll, pend.slot, pend_at);
      const uint32_t depth = __shfl_sync(kAll, pend.depth, pend_at) & kDepthMask;
      if (lane == q) my_slot = slot;
      if (lane < L) skeys[warp][q][lane] = __ldg(a.keys[depth & 1] + start + lane);
      if (lane == 0) {
        sdkey[warp][q] = uint64_t(depth) * kWeyl;
        sbase[warp][q] = 0;
        sbest[warp][q] = ~0u;
      }
      act |= 1u << q;
      pend_at++;
    }
    if (!act) break;
    __syncwarp();
    // the four quarters of the warp are dealt to the k slots in use: quarter
    // -> slot in order, the lanes on that slot, and the quarter's place among them
    const uint32_t k = __popc(act), quarter = lane >> 3;
    uint32_t mine = quarter, lanes = 8, place = 0;
    if (k < kPackedSlots) {
      const uint32_t rank = k == 3 ? (quarter == 3 ? 0 : quarter) : (k == 2 ? quarter & 1 : 0);
      mine = __fns(act, 0, static_cast<int>(rank) + 1);
      lanes = k == 1 ? 32 : (k == 2 || rank == 0 ? 16 : 8);
      place = k == 1 ? quarter : (k == 2 ? quarter >> 1 : quarter / 3);
    }
    uint64_t x[L];
#pragma unroll
    for (int j = 0; j < L; j++) x[j] = skeys[warp][mine][j];
    const uint64_t dkey = sdkey[warp][mine];
    uint32_t base = sbase[warp][mine];
    const uint32_t sub = 8 * place + (lane & 7);
    const uint64_t step = kWeyl64 * lanes;
    const uint32_t tag = mine << 16;
    // checked for equal keys in the first round at or beyond the stall point
    // (again if the lanes were dealt anew since: a round is 32 spl indices at most)
    uint32_t check = base < stall + 32 * kMaxSpl ? min(stall, limit) : limit;

    bool stop = false, won = false;
    while (!won) {
      if ((++rounds & 255) == 0 && __shfl_sync(kAll, lane == 0 ? *reinterpret_cast<volatile int*>(a.error) : 0, 0)) {
        stop = true;  // another search failed, or the host cancelled the build
        break;
      }
      if (__any_sync(kAll, base >= check)) {
        bool bad = false;
        if (base >= limit) {
          set_error(a.error, RECSPLIT_E_SEARCH_LIMIT);
          bad = true;
        } else if (base >= check) {
          check = limit;
          bool dup = false;
#pragma unroll
          for (int i = 0; i < L; i++)
#pragma unroll
            for (int j = i + 1; j < L; j++) dup |= x[i] == x[j];
          if (dup) set_error(a.error, RECSPLIT_E_DUPLICATE);
          bad = dup;
        }
        if (__any_sync(kAll, bad)) {
          stop = true;
          break;
        }
      }
      uint32_t ns = 0, idx = base + sub;
      uint64_t key = index_key(idx, dkey);
#pragma unroll 2
      for (uint32_t j = 0; j < spl; j++, key += step, idx += lanes) {
        if constexpr (kOne) {
          const uint64_t kp = key ^ (key >> 30);
          const bool ok = RANGE ? leaf_trial_range<L>(x, range, kp) : leaf_trial_full<L>(x, kp);
          if (ok) atomicMin(&sbest[warp][mine], idx);
          won |= __any_sync(kAll, ok);
        } else {
          uint32_t seen;
          const bool ok = leaf_head<L, H>(x, key ^ (key >> 30), reinterpret_cast<const uint8_t*>(lut), seen);
          const uint32_t b = __ballot_sync(kAll, ok);
          if (ok) surv[warp][ns + __popc(b & below)] = make_uint2(idx, seen | tag);
          ns += __popc(b);
        }
      }
      base += lanes * spl;
      __syncwarp();
      for (uint32_t t0 = 0; !kOne && t0 < ns; t0 += 32) {
        const uint32_t t = t0 + lane;
        bool ok = false;
        if (t < ns) {
          const uint2 e = surv[warp][t];
          const uint32_t s = e.y >> 16;
          const uint64_t ki = index_key(e.x, sdkey[warp][s]);
          const uint64_t kp = ki ^ (ki >> 30);
          uint32_t seen = e.y & 0xFFFFu;
#pragma unroll
          for (int i = H; i < L; i++) seen += 1u << phi_fixed<L>(skeys[warp][s][i], kp);
          ok = seen == full;
          if (ok) atomicMin(&sbest[warp][s], e.x);
        }
        won |= __any_sync(kAll, ok);
      }
      if (a.exec_count) exec += spl * 32 * H + ns * (L - H);
    }
    if (stop) break;
    __syncwarp();
    const uint32_t best = lane < kPackedSlots && (act >> lane & 1) ? sbest[warp][lane] : ~0u;
    if (best != ~0u) {
      a.seeds[my_slot] = best;
      a.sizes[my_slot] = L;
    }
    act &= ~__ballot_sync(kAll, best != ~0u);
    if (sub == 0) sbase[warp][mine] = base;
    __syncwarp();
  }
  if (a.exec_count && lane == 0 && exec) atomicAdd(a.exec_count, exec);
}

// Dynamic shared memory the split kernels may use: nodes of up to
// kSplitSmemBudget bytes of keys are staged, larger ones read from global
// memory; the tables of modes 8 and 9 come on top.
constexpr size_t kSplitSmemBudget = 96 * 1024;
constexpr size_t kSplitTableBytes = 2 * kPartCounts * sizeof(uint32_t);

// Raises the kernel's dynamic shared memory limit to the budget, once per
// kernel and process.  Setting it per launch to the launch's own size would
// race between builds on several host threads (the serving engine's
// workers): one thread could lower the limit between another's setting and
// its launch, which would then fail.
// (Once per kernel and device: KERNEL is the kernel itself, so every
// instantiation keeps flags of its own.)
template <auto KERNEL>
int allow_split_smem() {
  static std::once_flag once[64];
  static cudaError_t status[64] = {};
  int dev = 0;
  RS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(RECSPLIT_E_INVALID, "device ordinal above 63");
  std::call_once(once[dev], [&] {
    status[dev] = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        int(kSplitSmemBudget + kSplitTableBytes));
  });
  if (status[dev] != cudaSuccess) return cuda_fail(status[dev], "cudaFuncSetAttribute");
  return RECSPLIT_OK;
}

template <typename K>
int persistent_grid(K kernel, size_t smem, int sm_count, int* blocks) {
  int per_sm = 0;
  RS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, smem));
  if (per_sm < 1) return fail(RECSPLIT_E_INVALID, "search kernel does not fit on an SM");
  *blocks = per_sm * sm_count;
  return RECSPLIT_OK;
}

template <typename K, typename... Args>
int launch_persistent(K kern, int max_blocks, const SearchArgs& a, int sm_count, cudaStream_t s, Args... args) {
  int blocks = 0;
  int rc = persistent_grid(kern, 0, sm_count, &blocks);
  if (rc) return rc;
  kern<<<std::min(blocks, max_blocks), kThreads, 0, s>>>(a, args...);
  count_launch();
  RS_CUDA(cudaGetLastError());
  return RECSPLIT_OK;
}

// Leaves of 2 to L keys of a queue, each by the search for its size.
template <int L, bool RANGE>
int launch_any(const SearchArgs& a, const recsplit_tuning_t& t, int sm, cudaStream_t s, uint32_t qfull) {
  return launch_persistent(k_leaves<L, true, false, RANGE>, INT_MAX, a, sm, s, t.leaf_warps, t.leaf_chunk, 1u, qfull);
}

// Whether the packed kernel takes the class's full leaves of L keys.  The
// queue's capacity (keys / L + 1) bounds the leaves; with fewer than one per
// four warps of the grid (about four CTAs per SM) the two-phase kernel puts
// several warps on each.
template <int L>
bool packed_leaves(const SearchArgs& a, const recsplit_tuning_t& t, int sm) {
  return L >= 4 && L <= kPackedLeaf && t.leaf_two_phase && t.leaf_warps == 1 &&
         uint64_t(a.full_cap[a.cls]) > uint64_t(sm) * kWarps;
}

template <int L>
int launch_full(const SearchArgs& a, const recsplit_tuning_t& t, int sm, cudaStream_t s, const SharedNodes* share) {
  if constexpr (L >= kFifoLeaf) {
    if (t.leaf_two_phase && share)
      return launch_persistent(k_leaves_shared<L>, int(kSharedCtas), a, sm, s, *share, t.leaf_seeds_per_lane);
  } else {
    if constexpr (L >= 4 && L <= kPackedLeaf)
      if (packed_leaves<L>(a, t, sm))
        return launch_persistent(k_leaves_packed<L, false>, INT_MAX, a, sm, s, t.leaf_chunk, t.leaf_seeds_per_lane);
    if (t.leaf_two_phase)
      return launch_persistent(k_leaves<L, false, true>, INT_MAX, a, sm, s, t.leaf_warps, t.leaf_chunk,
                               t.leaf_seeds_per_lane, 1u);
  }
  return launch_persistent(k_leaves<L, false, false>, INT_MAX, a, sm, s, t.leaf_warps, t.leaf_chunk,
                           t.leaf_seeds_per_lane, 1u);
}

// Full leaves of the perfect, non-minimal variant.
template <int L>
int launch_full_range(const SearchArgs& a, const recsplit_tuning_t& t, int sm, cudaStream_t s, const SharedNodes*) {
  if constexpr (L >= 4 && L <= kPackedLeaf)
    if (packed_leaves<L>(a, t, sm))
      return launch_persistent(k_leaves_packed<L, true>, INT_MAX, a, sm, s, t.leaf_chunk, 1u);
  if (L <= 8) return launch_any<8, true>(a, t, sm, s, 1);
  if (L <= 16) return launch_any<16, true>(a, t, sm, s, 1);
  return launch_any<24, true>(a, t, sm, s, 1);
}

typedef int (*FullLauncher)(const SearchArgs&, const recsplit_tuning_t&, int, cudaStream_t, const SharedNodes*);
template <size_t... L>
constexpr auto full_launchers(std::index_sequence<L...>) {
  return std::array<FullLauncher, sizeof...(L) + 2>{nullptr, nullptr, launch_full<int(L) + 2>...};
}
template <size_t... L>
constexpr auto range_launchers(std::index_sequence<L...>) {
  return std::array<FullLauncher, sizeof...(L) + 2>{nullptr, nullptr, launch_full_range<int(L) + 2>...};
}
// by leaf size 2 .. kMaxLeaf
constexpr auto kFull = full_launchers(std::make_index_sequence<kMaxLeaf - 1>{});
constexpr auto kFullRange = range_launchers(std::make_index_sequence<kMaxLeaf - 1>{});

}  // namespace

// ---------------------------------------------------------------- tuning
namespace {
std::mutex g_tune_mu;
recsplit_tuning_t g_tune[kMaxLeaf + 1];
bool g_tuned[kMaxLeaf + 1] = {};
}  // namespace

// Seeds per lane that a leaf test mode starts from: one for the one-phase
// test; for the phased tests the fastest measured at each size (leaf phase,
// b = 100: l = 5: 1; l = 6: 2; l = 7, 8: 4; l = 9, 10: 8, 0.83 and 1.83 ms on 10^6
// keys against 0.85 and 1.90 with 4; from 12 keys a leaf takes thousands of
// trials and longer rounds spread the per-round checks).
uint32_t natural_seeds_per_lane(uint32_t leaf, uint32_t two_phase) {
  if (!two_phase) return 1;
  return leaf >= 9 ? kMaxSpl : (leaf >= 7 ? 4 : (leaf == 6 ? 2 : 1));
}

// (the phased tests are the faster from 4 keys on: leaf phase of 10^7 keys at
// l = 8, b = 100 3.4 ms with the one-phase test, 2.6 ms with the packed kernel)
recsplit_tuning_t default_tuning(uint32_t leaf) {
  recsplit_tuning_t t;
  t.leaf_warps = leaf >= 12 ? 4 : 1;
  t.leaf_chunk = leaf >= 12 ? 1 : 4;
  t.leaf_two_phase = leaf >= 4 ? 1 : 0;
  t.leaf_seeds_per_lane = natural_seeds_per_lane(leaf, t.leaf_two_phase);
  t.split_warps[0] = 1;
  t.split_warps[1] = leaf >= 12 ? 2 : 1;
  t.split_warps[2] = 8;
  return t;
}

recsplit_tuning_t tuning_for(uint32_t leaf) {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  if (leaf > kMaxLeaf || !g_tuned[leaf]) return default_tuning(leaf);
  return g_tune[leaf];
}

void set_tuning_for(uint32_t leaf, const recsplit_tuning_t& t) {
  std::lock_guard<std::mutex> lock(g_tune_mu);
  g_tune[leaf] = t;
  g_tuned[leaf] = true;
}

int launch_split_level(const SearchArgs& a, uint64_t max_m, uint64_t trials, uint32_t max_leaf, bool tables,
                       int sm_count, cudaStream_t s, const SharedNodes* share) {
  const size_t table_bytes = tables ? kSplitTableBytes : 0;
  if (share) {
    // one CTA per node at a time, nodes shared once the queue is empty
    const uint64_t cap = std::min<uint64_t>((max_m + 1) & ~uint64_t(1), kSplitSmemBudget / sizeof(uint64_t));
    const size_t smem = table_bytes + cap * sizeof(uint64_t);
    auto kern = a.exec_count ? k_split_shared<true> : k_split_shared<false>;
    int rc = a.exec_count ? allow_split_smem<k_split_shared<true>>() : allow_split_smem<k_split_shared<false>>();
    if (rc) return rc;
    int blocks = 0;
    rc = persistent_grid(kern, smem, sm_count, &blocks);
    if (rc) return rc;
    blocks = std::min<int>(blocks, kSharedCtas);
    kern<<<blocks, kThreads, smem, s>>>(a, *share, static_cast<uint32_t>(cap), uint32_t(tables));
    count_launch();
    RS_CUDA(cudaGetLastError());
    return RECSPLIT_OK;
  }
  // heavier nodes get more warps: fewer nodes per level and longer searches
  const recsplit_tuning_t t = tuning_for(max_leaf);
  const uint32_t gwarps = t.split_warps[max_m >= 256 ? 2 : (max_m >= 64 ? 1 : 0)];
  const uint32_t groups = kWarps / gwarps;
  // an even number of keys per group, so that every group's are 16-byte aligned
  const uint64_t cap = std::min<uint64_t>((max_m + 1) & ~uint64_t(1), kSplitSmemBudget / (groups * sizeof(uint64_t)));
  const size_t smem = table_bytes + size_t(groups) * cap * sizeof(uint64_t);
  auto kern = a.exec_count ? k_split_level<true> : k_split_level<false>;
  int rc = a.exec_count ? allow_split_smem<k_split_level<true>>() : allow_split_smem<k_split_level<false>>();
  if (rc) return rc;
  int blocks = 0;
  rc = persistent_grid(kern, smem, sm_count, &blocks);
  if (rc) return rc;
  kern<<<blocks, kThreads, smem, s>>>(a, gwarps, static_cast<uint32_t>(cap), uint32_t(tables), group_spread(trials));
  count_launch();
  RS_CUDA(cudaGetLastError());
  return RECSPLIT_OK;
}

bool leaves_shared(uint32_t leaf, uint32_t extra) {
  return !extra && leaf >= uint32_t(kFifoLeaf) && tuning_for(leaf).leaf_two_phase;
}

int launch_leaves(const SearchArgs& a, uint32_t leaf, uint32_t extra, uint64_t largest, int sm_count, cudaStream_t s,
                  const SharedNodes* share) {
  if (leaf < 2 || largest < 2) return RECSPLIT_OK;
  const recsplit_tuning_t t = tuning_for(leaf);
  // The kernels of full leaves read the table's entry of `leaf` keys whether or
  // not their queue is empty, so they are launched only where the table has it:
  // a class whose buckets are all smaller has no full leaf.
  int rc = largest >= leaf ? (extra ? kFullRange : kFull)[leaf](a, t, sm_count, s, share) : RECSPLIT_OK;
  if (rc || leaf == 2) return rc;  // no leaves between 2 and leaf - 1
  SearchArgs b = a;
  b.work_counter++;
  if (extra)
    return leaf <= 8    ? launch_any<8, true>(b, t, sm_count, s, 0)
           : leaf <= 16 ? launch_any<16, true>(b, t, sm_count, s, 0)
                        : launch_any<24, true>(b, t, sm_count, s, 0);
  return leaf <= 8    ? launch_any<8, false>(b, t, sm_count, s, 0)
         : leaf <= 12 ? launch_any<12, false>(b, t, sm_count, s, 0)
         : leaf <= 16 ? launch_any<16, false>(b, t, sm_count, s, 0)
                      : launch_any<24, false>(b, t, sm_count, s, 0);
}

}  // namespace rs
