// Lookup (Sec. 4, Sec. 6.2): signature -> bucket -> s_b, s_{b+1}, o_b from
// the double Elias-Fano lists (Sec. 6.3, Sec. 7.4) -> descent of the bucket's
// splitting tree.  At every split the key's part j is computed with the
// node's stored index; moving to child j skips the j earlier siblings, whose
// fixed parts are skipped with the table (a pointer move) and whose unary
// parts are skipped by counting j * codes(unit) ones; at the leaf the
// bijection's value is added to the keys left behind (c) and to s_b.
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "device.cuh"

namespace rs {
namespace {

// Sec. 6.3 / 7.4: o_b of bucket b, whose prefix s_b is s0, from the second Elias-Fano list.
__device__ __forceinline__ uint64_t ef_offset(const View& v, uint64_t b, uint64_t s0) {
  const uint64_t pb = ef_select(v, 1, b);
  const uint64_t xb = ((pb - b) << v.low_b) | read_bits(v.lower, b * (v.low_a + v.low_b) + v.low_a, v.low_b);
  const int64_t z = static_cast<int64_t>(xb) + static_cast<int64_t>(b) * v.delta_b;
  const uint64_t bs = (__umul64hi(s0, v.beta) << 32) | ((s0 * v.beta) >> 32);
  return static_cast<uint64_t>(z + static_cast<int64_t>(bs));
}

// Descent of a bucket of m >= 2 keys whose code starts at bit o.  RANGE: the
// structure has a leaf range extra (perfect, non-minimal variant); false
// compiles the minimal structure's path alone.
template <bool RANGE>
__device__ __forceinline__ uint64_t descend(const View& v, uint64_t s0, uint32_t m, uint64_t o, uint64_t lo);

// Output range of a subtree of m keys (table word 3, upper half).
__device__ __forceinline__ uint64_t node_range(const View& v, uint64_t m) {
  return __ldg(v.table + kTableWords * m + 3) >> 32;
}

// The bucket size whose output range is R.  Without a leaf range extra the
// range is the size; with one, ranges grow strictly with the size (the tables
// are built only then), so a binary search over sizes 0 .. mmax finds it.
template <bool RANGE>
__device__ __forceinline__ uint32_t size_of_range(const View& v, uint64_t R) {
  if (!RANGE || v.extra == 0) return static_cast<uint32_t>(R);
  uint64_t a = 0, b = v.mmax;
  while (a < b) {
    const uint64_t mid = (a + b + 1) >> 1;
    if (node_range(v, mid) <= R)
      a = mid;
    else
      b = mid - 1;
  }
  return static_cast<uint32_t>(a);
}

// Decoded buckets are {s_i | size << kSizeShift, o_i or a key}: values below 2^40,
// sizes below 2^24.
constexpr int kSizeShift = 40;
bool decode_fits(uint64_t range, uint64_t mmax) { return range < (1ull << kSizeShift) && mmax < (1ull << 24); }

// s_b and the size of bucket b (two consecutive elements of the first list).
template <bool RANGE>
__device__ __forceinline__ uint64_t bucket_start(const View& v, uint64_t b, uint32_t& m) {
  const uint32_t rec_w = v.low_a + v.low_b;
  const uint64_t rec = b * rec_w;
  const uint64_t pa = ef_select(v, 0, b);
  const uint64_t pa1 = next_one(v.upper_a, pa + 1);
  const uint64_t xa0 = ((pa - b) << v.low_a) | read_bits(v.lower, rec, v.low_a);
  const uint64_t xa1 = ((pa1 - b - 1) << v.low_a) | read_bits(v.lower, rec + rec_w, v.low_a);
  const uint64_t s0 = xa0 + static_cast<uint64_t>(static_cast<int64_t>(b) * v.delta_a);
  const uint64_t s1 = xa1 + static_cast<uint64_t>(static_cast<int64_t>(b + 1) * v.delta_a);
  m = size_of_range<RANGE>(v, s1 - s0);
  return s0;
}

template <bool RANGE>
__device__ __forceinline__ uint64_t lookup_one(const View& v, uint64_t hi, uint64_t lo) {
  if (v.nb == 0) return 0;
  const uint64_t b = bucket_of(hi, v.nb);
  uint32_t m;
  const uint64_t s0 = bucket_start<RANGE>(v, b, m);
  if (m <= 1) return s0;
  return descend<RANGE>(v, s0, m, ef_offset(v, b, s0), lo);
}

// Loads of what a decode launch before the lookup wrote.  The lookup's grid can
// start before that launch ends (launch_lookup), so these are neither read-only
// loads nor free to move above the wait for it.
__device__ __forceinline__ uint64_t load_decoded(const uint64_t* p) {
  uint64_t x;
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ ulonglong2 load_decoded(const ulonglong2* p) {
  ulonglong2 x;
  asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(x.x), "=l"(x.y) : "l"(p));
  return x;
}

// The same lookup with s_i, the size and o_i of every bucket decoded beforehand
// (decode_pays).
template <bool RANGE>
__device__ __forceinline__ uint64_t lookup_decoded(const View& v, const uint64_t* so, uint64_t hi,
                                                   uint64_t lo) {
  if (v.nb == 0) return 0;
  const uint64_t b = bucket_of(hi, v.nb);
  const ulonglong2 p = load_decoded(reinterpret_cast<const ulonglong2*>(so) + b);
  const uint64_t s0 = p.x & ((1ull << kSizeShift) - 1);
  const uint32_t m = static_cast<uint32_t>(p.x >> kSizeShift);
  if (m <= 1) return s0;
  return descend<RANGE>(v, s0, m, p.y, lo);
}

// Bit reads inside one bucket's code.  The tree bits are read as 32-bit
// little-endian words (bit k of the vector is bit k mod 32 of 32-bit word
// k / 32, the same bits as the 64-bit layout), with positions relative to the
// 32-bit word `t` that holds the code's first bit.  A bucket's code takes about
// two bits per key and the build rejects one that reaches 2^32 bits, so
// positions fit 32-bit registers.  32-bit words make every mask, shift, find
// and count a single instruction.  (64-bit words, half the loads but more
// instructions a level, were slower: from host call to end of 1000 queries, l = 12,
// b = 2000, 10^6 keys 22.4 us with 32-bit words and 23.0 with 64-bit ones, l = 8, b =
// 100 with a leaf range extra 19.3 and 19.6, without 17.1 and 17.2; 10^6 queries, l = 8,
// 10^7 keys 34.0 and 35.0, l = 12, 3 * 10^6 keys 35.1 and 37.1.  Only l = 5, b = 5, 10^7
// keys favours them: 3 * 10^5 queries 24.0 and 22.8, 10^6 55.5 and 55.0.)
//
// Scans stop at `end`, the 32-bit words from t to the end of the tree
// section, and then return 2^32 - 1: the structure check of deserialize
// already guarantees that every bucket's unary part holds its codes' one
// bits, so this only bounds the reads.
__device__ __forceinline__ uint32_t code_next_one(const uint32_t* __restrict__ t, uint32_t pos, uint32_t end) {
  uint32_t w = pos >> 5;
  uint32_t word = __ldg(t + w) & (~0u << (pos & 31));
  while (!word) {
    if (++w >= end) return ~0u;
    word = __ldg(t + w);
  }
  return (w << 5) + static_cast<uint32_t>(__ffs(word) - 1);
}

// Position of the set bit of rank k (0-based) in a 32-bit word (k < popc).
__device__ __forceinline__ uint32_t select_in_word32(uint32_t w, uint32_t k) {
  uint32_t pos = 0, c = __popc(w & 0xFFFFu);
  if (k >= c) { k -= c; pos = 16; w >>= 16; }
  c = __popc(w & 0xFFu);
  if (k >= c) { k -= c; pos += 8; w >>= 8; }
  c = __popc(w & 0xFu);
  if (k >= c) { k -= c; pos += 4; w >>= 4; }
  c = __popc(w & 0x3u);
  if (k >= c) { k -= c; pos += 2; w >>= 2; }
  return pos + (k >= (w & 1u) ? 1u : 0u);
}

__device__ __forceinline__ uint32_t code_select(const uint32_t* __restrict__ t, uint32_t pos, uint32_t rank,
                                                uint32_t end) {
  uint32_t w = pos >> 5;
  uint32_t word = __ldg(t + w) & (~0u << (pos & 31));
  for (;;) {
    const uint32_t c = __popc(word);
    if (rank < c) break;
    rank -= c;
    if (++w >= end) return ~0u;
    word = __ldg(t + w);
  }
  return (w << 5) + select_in_word32(word, rank);
}

// Position of the set bit of rank k (0-based) in a 64-bit word (k < popc).
__device__ __forceinline__ uint32_t select_in_word64(uint64_t x, uint32_t k) {
  const uint32_t lo = static_cast<uint32_t>(x);
  const uint32_t c = __popc(lo);
  const bool up = k >= c;
  return (up ? 32u : 0u) + select_in_word32(up ? static_cast<uint32_t>(x >> 32) : lo, up ? k - c : k);
}

// The 64 bits of the code from bit pos (relative to t), zero past `end`.
__device__ __forceinline__ uint64_t window64(const uint32_t* __restrict__ t, uint32_t pos, uint32_t end) {
  const uint32_t w = pos >> 5, sh = pos & 31;
  const uint32_t a0 = w < end ? __ldg(t + w) : 0u;
  const uint32_t a1 = w + 1 < end ? __ldg(t + w + 1) : 0u;
  const uint32_t a2 = w + 2 < end ? __ldg(t + w + 2) : 0u;
  return (uint64_t(__funnelshift_r(a1, a2, sh)) << 32) | __funnelshift_r(a0, a1, sh);
}

// (i * 64 + d) * W = i * (64 W) + d * W: the family key of index i at depth d
// as one multiply-add, the depth term advancing by W per level.
constexpr uint64_t kWeyl64 = kWeyl << 6;

// Sec. 4 / 6.2: descent of the splitting tree of a bucket of m >= 2 keys
// whose code starts at bit o.  Per node of m keys
// one 16-byte lookup record gives r, the fanout, the part size, the
// reciprocal for the part index, and the fixed bits and codes of a part-sized
// subtree (to skip the earlier siblings).  The unary part of the bucket's
// code (one code per node, about 1.5 bits each) is held in a 64-bit register
// window from its first bit, so reading a unary code is a find-first-set and
// skipping j * codes(unit) codes a select inside the window.  Where the
// window runs out (buckets of thousands of keys), a scan of the code words
// finds the position and the window is reloaded there: the chosen subtree's
// codes follow it, so the rest of the descent reads the new window.  Fixed parts
// are read with two loads and a funnel shift, without a branch.  With a leaf
// range extra e (RANGE), a leaf of m keys maps into m + e values and the
// siblings left behind contribute their output ranges (table word 3) instead
// of their keys.
template <bool RANGE>
__device__ __forceinline__ uint64_t descend(const View& v, uint64_t s0, uint32_t m, uint64_t o, uint64_t lo) {
  const uint32_t* __restrict__ t = reinterpret_cast<const uint32_t*>(v.tree) + (o >> 5);
  const uint64_t left = v.tree_words32 - (o >> 5);
  const uint32_t end = left < 0xFFFFFFFFull ? static_cast<uint32_t>(left) : 0xFFFFFFFFu;
  uint32_t fixed = static_cast<uint32_t>(o & 31);
  // the unary part starts after the fixed parts of all the bucket's codes
  const uint32_t u0 = fixed + static_cast<uint32_t>(__ldg(v.table + kTableWords * m));
  uint32_t wb = 0;  // first bit of the window, relative to u0
  uint64_t win = window64(t, u0, end);
  uint32_t up = 0;  // bit of the next unary code, relative to u0
  const uint64_t xpre = pre_key(lo);
  uint64_t dkey = 0;  // depth * W
  uint32_t c = 0;     // keys of the siblings left behind
  const uint4* __restrict__ rec = reinterpret_cast<const uint4*>(v.rec);
  uint4 nd = __ldg(rec + m);
  for (;;) {
    const uint32_t r = (nd.w >> kLookupCodeBits) & 31, fanout = nd.w >> 28;
    const uint32_t fw = fixed >> 5;
    const uint32_t f0 = __ldg(t + fw);
    const uint32_t f1 = fw + 1 < end ? __ldg(t + fw + 1) : 0u;
    const uint32_t low = __funnelshift_r(f0, f1, fixed & 31) & ((1u << r) - 1u);
    fixed += r;
    const uint32_t rel = up - wb;
    const uint64_t rest = rel < 64 ? win >> rel : 0ull;
    uint32_t one;  // the unary code's one bit, relative to u0
    if (rest) {
      one = up + static_cast<uint32_t>(__ffsll(static_cast<long long>(rest)) - 1);
    } else {
      const uint32_t a = code_next_one(t, u0 + up, end);
      if (a == ~0u) return ~0ull;
      one = a - u0;
      wb = one;  // the rest of the descent reads from here on
      win = window64(t, u0 + wb, end);
    }
    const uint64_t seed = (uint64_t(one - up) << r) | low;
    up = one + 1;
    const uint64_t k = seed * kWeyl64 + dkey;
    const uint32_t h = family_top32(xpre, k ^ (k >> 30));
    if (fanout == 0) return s0 + c + __umulhi(h, RANGE ? m + v.extra : m);
    const uint32_t val = __umulhi(h, m);
    const uint32_t part = min(nd.y ? __umulhi(val, nd.y) : val / nd.x, fanout - 1);
    if (part) {
      fixed += part * nd.z;
      // skip the unary codes of the part earlier siblings (none when a
      // part-sized subtree has no code, e.g. single keys): up moves past the
      // one of rank part * codes(unit) - 1
      const uint32_t skip = part * (nd.w & ((1u << kLookupCodeBits) - 1));
      if (skip) {
        const uint32_t rel = up - wb;
        const uint64_t x = rel < 64 ? win & (~0ull << rel) : 0ull;
        if (static_cast<uint32_t>(__popcll(x)) >= skip) {
          up = wb + select_in_word64(x, skip - 1) + 1;
        } else {
          const uint32_t a = code_select(t, u0 + up, skip - 1, end);
          if (a == ~0u) return ~0ull;
          up = a - u0 + 1;
          wb = up;  // the chosen subtree's codes start here
          win = window64(t, u0 + wb, end);
        }
      }
      // keys (or, with a leaf range extra, output ranges) of the siblings left behind
      c += RANGE ? static_cast<uint32_t>(part * node_range(v, nd.x)) : part * nd.x;
    }
    m = part + 1 < fanout ? nd.x : m - nd.x * (fanout - 1);
    if (m <= 1) return s0 + c;
    nd = __ldg(rec + m);
    dkey += kWeyl;
  }
}

// ---------------------------------------------------------------- flat codes
// A batch of at least 1.5 queries per code of the structure (flat_pays) decodes every
// code once: the function key K ^ (K >> 30) of code c (preorder) of bucket b is stored
// at place flat_base(s_b, b) + c, and so holds s_b, the bucket's size and the key of its
// first code in 16 bytes: {s_b | m << 40, key}.  A level of the
// descent then loads its key and steps over the earlier siblings' codes with
// one multiply-add, where it otherwise reads a fixed part, finds a unary part
// and selects past the siblings in the bit vector.
//
// A bucket of m keys has at most rho m + 3 codes, rho = 1 / l + 1 / lower + 2 / upper (a leaf
// and a node of each kind per so many keys, two at the top, and of each kind at
// most one that is not full), and fewer than m, so the places floor(rho s_b) + 4 b .. of
// different buckets are disjoint and nearly all are used: the keys of a lookup's
// level share sectors.
// (One place per value of the range: 4 * 10^7 keys, l = 8, b = 100, three queries per
// code 0.69 ms against 0.38; 3.4 * 10^7 keys in 256 structures, 7 * 10^7 queries 2.7
// against 1.9 ms.)
constexpr uint32_t kFlatSlack = 4;  // places per bucket beyond rho s_b

// rho in units of 2^-32 (below 1: a bucket has fewer codes than keys), by leaf size: a table,
// since a batch asks for it per structure.
struct FlatSlopes {
  uint32_t of[kMaxLeaf + 1];
  FlatSlopes() : of{} {
    for (uint32_t leaf = 1; leaf <= kMaxLeaf; leaf++) {
      const Strategy st = make_strategy(leaf);
      uint64_t slope = 0;
      for (uint64_t u : {uint64_t(st.leaf), st.lower, st.upper, st.upper}) slope += ((1ull << 32) + u - 1) / u;
      of[leaf] = static_cast<uint32_t>(std::min<uint64_t>(slope, 0xFFFFFFFFull));
    }
  }
};
uint32_t flat_slope(uint32_t leaf) {
  static const FlatSlopes slopes;
  return slopes.of[leaf];
}

// Places of a structure; with at most kFlatPlaces of them s_b, b and the places fit
// 32 bits (rho is at least 1 / 24).
uint64_t flat_places(const Handle& h) {
  const uint64_t range = std::min<uint64_t>(h.range_size, 1ull << 40), nb = std::min<uint64_t>(h.header[H_NB], 1ull << 40);
  const uint64_t slope = flat_slope(header_leaf(h.header));
  const uint64_t high = (range >> 16) * slope, low = (range & 0xFFFF) * slope;  // range * slope in halves
  return (high >> 16) + (low >> 32) + 1 + kFlatSlack * nb;
}

__device__ __forceinline__ uint32_t flat_base(uint32_t slope, uint64_t s, uint64_t b) {
  return __umulhi(static_cast<uint32_t>(s), slope) + kFlatSlack * static_cast<uint32_t>(b);
}

// Key of code c of a bucket of m keys (fixed parts from bit `fixed` of t, unary
// part un): the path to node c of the preorder gives its size, depth and the
// position of its fixed part.
__device__ __forceinline__ uint64_t code_key(const View& v, const uint32_t* __restrict__ t, uint32_t end,
                                             uint32_t fixed, uint32_t m, uint32_t c, uint32_t un) {
  const uint4* __restrict__ rec = reinterpret_cast<const uint4*>(v.rec);
  uint32_t depth = 0, r;
  for (;;) {
    const uint4 nd = __ldg(rec + m);
    r = (nd.w >> kLookupCodeBits) & 31;
    if (c == 0) break;
    c--;
    const uint32_t codes = nd.w & ((1u << kLookupCodeBits) - 1), fanout = nd.w >> 28;
    const uint32_t j = codes ? min(c / codes, fanout - 1) : fanout - 1;
    c -= j * codes;
    fixed += r + j * nd.z;
    m = j + 1 < fanout ? nd.x : m - nd.x * (fanout - 1);
    depth++;
  }
  const uint32_t w = fixed >> 5;
  const uint32_t f0 = __ldg(t + w), f1 = w + 1 < end ? __ldg(t + w + 1) : 0u;
  const uint32_t low = __funnelshift_r(f0, f1, fixed & 31) & ((1u << r) - 1u);
  return family_key((uint64_t(un) << r) | low, depth);
}

// What the decode of the codes reads of a structure.
struct DecodeView : View {
  uint64_t* flat;      // function key of every code
  uint32_t slope;      // flat_slope
  uint32_t log_group;  // parts that a bucket's codes are decoded in, log2
};

// Part p of the decode of the structure's buckets, 2^log_group to a bucket: part g
// of bucket b decodes codes g, g + 2^log_group, ...  Every part reads the lists for
// itself and scans the unary part with a cursor of its own, so parts need
// nothing from each other.
template <bool RANGE>
__device__ __forceinline__ void flat_part(const DecodeView& v, uint64_t p) {
  const uint32_t log_group = v.log_group;
  const uint64_t b = p >> log_group;
  const uint32_t g = p & ((1u << log_group) - 1);
  if (b >= v.nb) return;
  uint64_t* so = const_cast<uint64_t*>(v.so);
  uint32_t m;
  const uint64_t s0 = bucket_start<RANGE>(v, b, m);
  if (g == 0) so[2 * b] = s0 | (uint64_t(m) << kSizeShift);
  if (m < 2) return;
  const uint64_t w0 = __ldg(v.table + kTableWords * m);
  const uint32_t codes = static_cast<uint32_t>(w0 >> 32);
  if (g >= codes) return;
  const uint64_t o = ef_offset(v, b, s0);
  const uint32_t* __restrict__ t = reinterpret_cast<const uint32_t*>(v.tree) + (o >> 5);
  const uint64_t left = v.tree_words32 - (o >> 5);
  const uint32_t end = left < 0xFFFFFFFFull ? static_cast<uint32_t>(left) : 0xFFFFFFFFu;
  const uint32_t fixed = static_cast<uint32_t>(o & 31);
  uint64_t* flat = v.flat + flat_base(v.slope, s0, b);
  const uint32_t u0 = fixed + static_cast<uint32_t>(w0);  // first bit of the unary part
  // cursor: `rank` ones lie in [u0, word w), `word` holds the ones of word w
  // from u0 on
  uint32_t w = u0 >> 5, rank = 0;
  uint32_t word = __ldg(t + w) & (~0u << (u0 & 31));
  for (uint32_t c = g; c < codes; c += 1u << log_group) {
    uint32_t from = u0;  // the bit after the one of code c - 1
    if (c) {
      uint32_t ones = __popc(word);
      while (rank + ones < c) {
        if (++w >= end) return;
        rank += ones;
        word = __ldg(t + w);
        ones = __popc(word);
      }
      from = (w << 5) + select_in_word32(word, c - 1 - rank) + 1;
    }
    const uint32_t one = code_next_one(t, from, end);
    if (one == ~0u) return;
    const uint64_t key = code_key(v, t, end, fixed, m, c, one - from);
    flat[c] = key;
    if (c == 0) so[2 * b + 1] = key;
  }
}

// Parts (log2) that the buckets of a structure are decoded in, `per` codes or
// more to a part on average.  One thread per bucket left 10^4 buckets of 18
// codes waiting on dependent loads (13 us).
uint32_t flat_log_group(uint64_t codes, uint64_t nb, uint64_t per) {
  uint32_t lg = 0;
  while (lg < 10 && codes >= (nb * per) << (lg + 1)) lg++;
  return lg;
}

// Codes per part: two, or as many as keep all parts to 2^19 (about the
// threads the device holds).
uint64_t codes_per_part(uint64_t codes) { return std::max<uint64_t>(2, codes >> 19); }

// v (with so set) for a decode of the codes into `flat`, `per` codes or more to a part.
DecodeView decode_view(const Handle& h, const View& v, uint64_t* flat, uint64_t per) {
  DecodeView d;
  static_cast<View&>(d) = v;
  d.flat = flat;
  d.slope = flat_slope(header_leaf(h.header));
  d.log_group = v.nb ? flat_log_group(h.ncodes, v.nb, per) : 0;
  return d;
}

// Most places of the flat keys, 128 MiB: beyond, they are read from HBM, while the code bits of the
// same structures stay in L2.  l = 8, b = 100, three queries per code, lists alone and codes:
// 4 * 10^7 keys (70 MB of flat keys) 0.52 and 0.38 ms, 10^8 (174 MB) 1.26 and 1.35,
// 3 * 10^8 4.1 and 7.1.
constexpr uint64_t kFlatPlaces = 1ull << 24;

// Whether a batch of q queries decodes the codes first, at 1.5 queries per code: l =
// 8, b = 100, 10^7 keys (1.78 * 10^6 codes), with the lists decoded alone and with the
// codes: 1.0 queries per code 53 and 58 us, 1.5 73 and 70, 3.0 135 and 105; l = 12, b =
// 2000, 3 * 10^6 keys: 1.5 45 and 27 us.  Below 200000 queries the two paths are equal
// within 3 us, and buckets of a few codes have nothing to skip (l = 5, b = 5: 1.6 codes,
// 517 us without and 546 with it for ten queries per code).
bool flat_pays(uint64_t q, uint64_t codes, uint64_t nb, uint64_t places) {
  return places <= kFlatPlaces && 2 * q >= 3 * codes && q >= kDecodeQueries && codes >= 2 * nb;
}

// Whether a batch of q queries decodes the buckets of the lists first.  From host
// call to end, without the decode and with it:
//   one structure, l = 8, b = 100, 1000 buckets: 2 * 10^5 queries 23.4 and 24.9 us,
//     2.6 * 10^5 26.7 and 26.1, 4 * 10^5 31.8 and 28.6; 10^5 buckets 24.4 and 25.5, 29.4 and
//     26.8, 33.4 and 30.4; 1000 with a leaf range extra 24.8 and 26.1, 28.3 and 27.3, 34.0
//     and 30.2; l = 5, b = 5, 10^6 buckets: 4 * 10^5 33.3 and 40.5, 7 * 10^5 46.1 and 44.9;
//   40 structures, l = 8, b = 100, 100 buckets each: 2 * 10^5 37.2 and 39.8, 4 * 10^5 47.4
//     and 46.9, 7 * 10^5 60.4 and 53.7; 2500 each: 2.6 * 10^5 42.6 and 43.0, 4 * 10^5 53.6 and
//     48.9.
bool decode_pays(uint64_t q, uint64_t nb) { return q >= nb / 2 + (1u << 18); }

// What a flat lookup reads of a structure (16-byte loads where it is read per
// query).
struct alignas(16) FlatView {
  const ulonglong2* so;
  const uint64_t* flat;
  uint64_t nb;
  const uint64_t* table;  // output ranges (RANGE)
  // sizes of the splitting strategy (Sec. 5.4), their reciprocals ceil(2^32 / u)
  // and the codes of subtrees of `lower` and `upper` keys
  uint32_t leaf, lower, upper, leaf_magic;
  uint32_t lower_magic, upper_magic, lower_codes, upper_codes;
  const uint4* rec;
  uint32_t extra, slope;
};

FlatView flat_view(const Handle& h, const DecodeView& v) {
  const uint32_t leaf = header_leaf(h.header);
  const Strategy st = make_strategy(leaf);
  auto magic = [](uint64_t u) { return static_cast<uint32_t>(((1ull << 32) + u - 1) / u); };
  const uint32_t lower_codes = static_cast<uint32_t>(1 + st.lower / st.leaf);
  return FlatView{reinterpret_cast<const ulonglong2*>(v.so), v.flat, v.nb, v.table, leaf,
                  static_cast<uint32_t>(st.lower), static_cast<uint32_t>(st.upper),
                  leaf >= 2 ? magic(st.leaf) : 0, magic(st.lower), magic(st.upper), lower_codes,
                  static_cast<uint32_t>(1 + st.upper / st.lower * lower_codes),
                  reinterpret_cast<const uint4*>(v.rec), v.extra, v.slope};
}

template <bool RANGE>
__global__ void __launch_bounds__(256) k_flat_decode(const __grid_constant__ DecodeView v) {
  cudaTriggerProgrammaticLaunchCompletion();
  flat_part<RANGE>(v, blockIdx.x * uint64_t(blockDim.x) + threadIdx.x);
}

// Buckets of every structure: part p of the global index space belongs to the
// structure i with base[i] <= p < base[i + 1].
__global__ void __launch_bounds__(256) k_flat_decode_views(const DecodeView* __restrict__ views,
                                                           const uint64_t* __restrict__ base, uint32_t count,
                                                           uint64_t total) {
  const uint64_t p = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x;
  if (p >= total) return;
  uint32_t lo = 0, hi = count;  // last i with base[i] <= p
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) / 2;
    if (__ldg(base + mid) <= p) lo = mid; else hi = mid;
  }
  flat_part<true>(views[lo], p - __ldg(base + lo));
}

// Whether the steps of a descent can be computed (lookup_flat): the
// reciprocals are exact for values below 2^16, and leaves of one key have no
// code.
bool steps_computed(const Handle& h) { return h.header[H_MMAX] < 65536 && header_leaf(h.header) >= 2; }

// STEPS: the part, its size and the codes to step over are computed from the
// strategy's sizes instead of loaded by node size.  About 12 instructions
// replace a load that is scattered over the lanes: 64-bit keys, which are bound
// by such loads, gain (l = 8, b = 100, ten queries per code 280 -> 266 us; l = 12,
// b = 2000 85 -> 73 us; 256 structures 355 -> 319 us), strings, whose signatures
// keep the ALU pipe busy, lose (1.91 against 1.94 ms) and load.
template <bool RANGE, bool STEPS>
__device__ __forceinline__ uint64_t lookup_flat(const FlatView& v, uint64_t hi, uint64_t lo) {
  if (v.nb == 0) return 0;
  const uint64_t b = bucket_of(hi, v.nb);
  const ulonglong2 p = load_decoded(v.so + b);
  const uint64_t s0 = p.x & ((1ull << kSizeShift) - 1);
  uint32_t m = static_cast<uint32_t>(p.x >> kSizeShift);
  if (m <= 1) return s0;
  const uint64_t* code = v.flat + flat_base(v.slope, s0, b);
  const uint64_t xpre = pre_key(lo);
  uint32_t c = 0;  // keys (or output ranges) of the siblings left behind
  for (uint64_t kp = p.y;; kp = load_decoded(code)) {
    const uint32_t h = family_top32(xpre, kp);
    uint32_t unit, codes, part;  // of every child but the last; the key's child
    if constexpr (STEPS) {
      if (m <= v.leaf) return s0 + c + __umulhi(h, RANGE ? m + v.extra : m);
      const uint32_t val = __umulhi(h, m);
      const bool low = m <= v.lower;
      unit = low ? v.leaf : v.lower;
      codes = low ? 1u : v.lower_codes;
      part = __umulhi(val, low ? v.leaf_magic : v.lower_magic);
      if (m > v.upper) {
        // two children, the first of k * upper keys: k subtrees of `upper` under
        // k - 1 binary splits
        const uint32_t k = __umulhi((m >> 1) + v.upper - 1, v.upper_magic);
        unit = k * v.upper;
        codes = k * v.upper_codes + k - 1;
        part = val >= unit;
        m = part ? m - unit : unit;
      } else {
        m = min(unit, m - part * unit);
      }
    } else {
      const uint4 nd = __ldg(v.rec + m);
      const uint32_t fanout = nd.w >> 28;
      if (fanout == 0) return s0 + c + __umulhi(h, RANGE ? m + v.extra : m);
      const uint32_t val = __umulhi(h, m);
      unit = nd.x;
      codes = nd.w & ((1u << kLookupCodeBits) - 1);
      part = min(nd.y ? __umulhi(val, nd.y) : val / nd.x, fanout - 1);
      m = part + 1 < fanout ? unit : m - unit * (fanout - 1);
    }
    code += 1 + part * codes;
    c += RANGE ? part * static_cast<uint32_t>(__ldg(v.table + kTableWords * unit + 3) >> 32) : part * unit;
    if (m <= 1) return s0 + c;
  }
}

template <bool RANGE, bool STEPS>
__global__ void __launch_bounds__(256, 8) k_lookup_u64_flat(FlatView v, const uint64_t* __restrict__ keys, uint64_t q,
                                                            uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    uint64_t hi, lo;
    signature_u64(__ldg(keys + i), hi, lo);
    cudaGridDependencySynchronize();  // the decode's results are read from here on
    out[i] = lookup_flat<RANGE, STEPS>(v, hi, lo);
  }
}

template <bool RANGE>
__global__ void __launch_bounds__(256, 8) k_lookup_bytes_flat(FlatView v, const uint8_t* __restrict__ bytes,
                                                              const uint64_t* __restrict__ offsets, uint64_t q,
                                                              uint64_t* __restrict__ out) {
  const uint64_t last = __ldg(offsets + q);  // the bytes span [0, offsets[q])
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t o0 = __ldg(offsets + i), o1 = __ldg(offsets + i + 1);
    uint64_t hi, lo;
    const bool ok = o0 <= o1 && o1 <= last;  // else read as the empty string
    signature_bytes(bytes + (ok ? o0 : 0), ok ? o1 - o0 : 0, hi, lo);
    cudaGridDependencySynchronize();
    out[i] = lookup_flat<RANGE, false>(v, hi, lo);
  }
}

template <bool ANY_RANGE, bool STEPS>
__global__ void __launch_bounds__(256, 8) k_lookup_many_flat(const FlatView* __restrict__ views, uint32_t count,
                                                             const uint32_t* __restrict__ ids,
                                                             const uint64_t* __restrict__ keys, uint64_t q,
                                                             uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t id = __ldg(ids + i);
    if (id >= count) {
      out[i] = ~0ull;
      continue;
    }
    uint64_t hi, lo;
    signature_u64(__ldg(keys + i), hi, lo);
    const FlatView v = views[id];
    out[i] = ANY_RANGE && v.extra ? lookup_flat<true, STEPS>(v, hi, lo) : lookup_flat<false, STEPS>(v, hi, lo);
  }
}

template <bool RANGE>
__device__ __forceinline__ void decode_bucket(const View& v, uint64_t b) {
  uint64_t* so = const_cast<uint64_t*>(v.so);
  uint32_t m;
  const uint64_t s0 = bucket_start<RANGE>(v, b, m);
  reinterpret_cast<ulonglong2*>(so)[b] = make_ulonglong2(s0 | (uint64_t(m) << kSizeShift), ef_offset(v, b, s0));
}

// Every bucket, one thread each.
template <bool RANGE>
__global__ void k_ef_decode(View v) {
  cudaTriggerProgrammaticLaunchCompletion();
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < v.nb; i += uint64_t(gridDim.x) * blockDim.x)
    decode_bucket<RANGE>(v, i);
}

template <bool RANGE, bool DECODED>
__global__ void __launch_bounds__(256) k_lookup_u64(View v, const uint64_t* so, const uint64_t* __restrict__ keys,
                                                    uint64_t q, uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    uint64_t hi, lo;
    signature_u64(__ldg(keys + i), hi, lo);
    if (DECODED) cudaGridDependencySynchronize();  // the decode's results are read from here on
    out[i] = DECODED ? lookup_decoded<RANGE>(v, so, hi, lo) : lookup_one<RANGE>(v, hi, lo);
  }
}

// 32 registers (8 blocks of 256 threads per SM): the kernel is bound by
// instruction issue, and full occupancy outweighs a few spilled registers
// (measured: 4.09 -> 4.01 ms for 10^8 string lookups).
template <bool RANGE, bool DECODED>
__global__ void __launch_bounds__(256, 8) k_lookup_bytes(View v, const uint64_t* so,
                                                         const uint8_t* __restrict__ bytes,
                                                         const uint64_t* __restrict__ offsets, uint64_t q, uint64_t* __restrict__ out) {
  const uint64_t last = __ldg(offsets + q);  // the bytes span [0, offsets[q])
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint64_t o0 = __ldg(offsets + i), o1 = __ldg(offsets + i + 1);
    uint64_t hi, lo;
    const bool ok = o0 <= o1 && o1 <= last;  // else read as the empty string
    signature_bytes(bytes + (ok ? o0 : 0), ok ? o1 - o0 : 0, hi, lo);
    if (DECODED) cudaGridDependencySynchronize();
    out[i] = DECODED ? lookup_decoded<RANGE>(v, so, hi, lo) : lookup_one<RANGE>(v, hi, lo);
  }
}

// Buckets of every structure: bucket g of the global index space belongs to the
// structure i with base[i] <= g < base[i + 1].
__global__ void k_ef_decode_views(const View* __restrict__ views, const uint64_t* __restrict__ base, uint32_t count,
                                  uint64_t total) {
  for (uint64_t g = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; g < total; g += uint64_t(gridDim.x) * blockDim.x) {
    uint32_t lo = 0, hi = count;  // last i with base[i] <= g
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) / 2;
      if (__ldg(base + mid) <= g) lo = mid; else hi = mid;
    }
    const View& v = views[lo];
    decode_bucket<true>(v, g - __ldg(base + lo));
  }
}

// ANY_RANGE: some structure of the batch has a leaf range extra.  Bounded to
// 32 registers like k_lookup_bytes (measured: 10.0 -> 8.6 ms per 10^8
// batched lookups over 4096 structures).  A query whose structure id is not
// below `count` gets the value 2^64 - 1 (no structure is read for it).
// DECODED: the lists of every structure are decoded.  (Both lookups in one kernel
// spilled 64 and reloaded 104 bytes, the lookup without decoded lists alone 40 and
// 64: with the smaller views, 10^4 queries over 40 structures of 1000 buckets 25.9 ->
// 24.9 us.)
template <bool ANY_RANGE, bool DECODED>
__global__ void __launch_bounds__(256, 8) k_lookup_many(const View* __restrict__ views, uint32_t count,
                              const uint32_t* __restrict__ ids, const uint64_t* __restrict__ keys, uint64_t q,
                              uint64_t* __restrict__ out) {
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t id = __ldg(ids + i);
    if (id >= count) {
      out[i] = ~0ull;
      continue;
    }
    uint64_t hi, lo;
    signature_u64(__ldg(keys + i), hi, lo);
    const View& v = views[id];
    if constexpr (DECODED)
      out[i] = ANY_RANGE && v.extra ? lookup_decoded<true>(v, v.so, hi, lo) : lookup_decoded<false>(v, v.so, hi, lo);
    else
      out[i] = ANY_RANGE && v.extra ? lookup_one<true>(v, hi, lo) : lookup_one<false>(v, hi, lo);
  }
}

// (The serving engine's: it decodes nothing.)
__global__ void k_lookup_many_bytes(const View* __restrict__ views, uint32_t count, const uint32_t* __restrict__ ids,
                                    const uint8_t* __restrict__ bytes, const uint64_t* __restrict__ offsets,
                                    uint64_t q, uint64_t* __restrict__ out) {
  const uint64_t last = __ldg(offsets + q);  // the bytes span [0, offsets[q])
  for (uint64_t i = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x; i < q; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t id = __ldg(ids + i);
    if (id >= count) {
      out[i] = ~0ull;
      continue;
    }
    const uint64_t o0 = __ldg(offsets + i), o1 = __ldg(offsets + i + 1);
    uint64_t hi, lo;
    const bool ok = o0 <= o1 && o1 <= last;  // else read as the empty string
    signature_bytes(bytes + (ok ? o0 : 0), ok ? o1 - o0 : 0, hi, lo);
    const View& v = views[id];
    out[i] = v.extra ? lookup_one<true>(v, hi, lo) : lookup_one<false>(v, hi, lo);
  }
}

}  // namespace

// NVTX range around the launches of one lookup call.
struct LookupRange {
  LookupRange() { nvtxRangePushA("recsplit.lookup"); }
  ~LookupRange() { nvtxRangePop(); }
};

int lookup_many_bytes(const View* d_views, uint32_t count, const uint32_t* d_ids, const uint8_t* d_bytes,
                      const uint64_t* d_offsets, uint64_t q, uint64_t* d_out, cudaStream_t s) {
  if (q == 0) return RECSPLIT_OK;
  LookupRange range;
  int dev = 0, sms = 0;
  RS_CUDA(cudaGetDevice(&dev));
  RS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int block = 256;
  const uint64_t want = (q + block - 1) / block;
  const unsigned grid = static_cast<unsigned>(want < uint64_t(sms) * 64 ? want : uint64_t(sms) * 64);
  k_lookup_many_bytes<<<grid, block, 0, s>>>(d_views, count, d_ids, d_bytes, d_offsets, q, d_out);
  count_launch();
  RS_CUDA(cudaGetLastError());
  return RECSPLIT_OK;
}

int lookup_many(const View* d_views, uint32_t count, const uint32_t* d_ids, const uint64_t* d_keys, uint64_t q,
                uint64_t* d_out, cudaStream_t s, bool any_range, const FlatBatch* flat) {
  if (q == 0) return RECSPLIT_OK;
  LookupRange range;
  int dev = 0, sms = 0;
  RS_CUDA(cudaGetDevice(&dev));
  RS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int block = 256;
  const uint64_t want = (q + block - 1) / block;
  const unsigned grid = static_cast<unsigned>(want < uint64_t(sms) * 64 ? want : uint64_t(sms) * 64);
  if (flat && flat->views) {
    auto kern = flat->steps ? (any_range ? k_lookup_many_flat<true, true> : k_lookup_many_flat<false, true>)
                            : (any_range ? k_lookup_many_flat<true, false> : k_lookup_many_flat<false, false>);
    kern<<<grid, block, 0, s>>>(static_cast<const FlatView*>(flat->views), count, d_ids, d_keys, q, d_out);
  } else {
    auto kern = flat && flat->decoded ? (any_range ? k_lookup_many<true, true> : k_lookup_many<false, true>)
                                      : (any_range ? k_lookup_many<true, false> : k_lookup_many<false, false>);
    kern<<<grid, block, 0, s>>>(d_views, count, d_ids, d_keys, q, d_out);
  }
  count_launch();
  RS_CUDA(cudaGetLastError());
  return RECSPLIT_OK;
}

int decode_views(const Handle* const* hs, View* views, uint32_t count, uint64_t q, cudaStream_t s, uint64_t** scratch,
                 FlatBatch* batch) {
  *scratch = nullptr;
  *batch = FlatBatch{};
  if (q < kDecodeQueries) return RECSPLIT_OK;
  // the buckets of every structure, or their parts
  uint64_t buckets = 0, codes = 0, places = 0;
  bool fits = true, steps = true;
  for (uint32_t i = 0; i < count; i++) {
    buckets += views[i].nb;
    codes += hs[i]->ncodes;
    places += flat_places(*hs[i]);
    fits &= decode_fits(hs[i]->range_size, views[i].mmax);
    steps &= steps_computed(*hs[i]);
  }
  // Codes as well as lists are decoded from the lists' line on, later than for one
  // structure: 40 structures of 100 buckets, l = 8, b = 100: 2.5 * 10^5 queries, below the
  // line, 32.4 us, 3 * 10^5, with decoded codes, 32.7; of 20 buckets, l = 12, b = 2000:
  // 43.7 and 38.8.
  if (buckets == 0 || !decode_pays(q, buckets) || !fits) return RECSPLIT_OK;
  bool flat = flat_pays(q, codes, buckets, places);
  // one allocation: the views, the flat views, the first part of every view (one
  // copy), then the decoded buckets and, with the codes, their keys
  constexpr uint64_t kViewWords = sizeof(View) / 8, kDecodeWords = sizeof(DecodeView) / 8,
                     kFlatWords = sizeof(FlatView) / 8;
  static_assert(sizeof(View) % 8 == 0 && sizeof(DecodeView) % 8 == 0 && sizeof(FlatView) % 16 == 0,
                "views are copied as words");
  auto flat_at = [&] { return (count * (flat ? kDecodeWords : kViewWords) + 1) & ~uint64_t(1); };  // 16-byte aligned
  auto base_at = [&] { return flat_at() + (flat ? count * kFlatWords : 0); };
  auto so_at = [&] { return (base_at() + count + 2) & ~uint64_t(1); };
  void* d_scratch = nullptr;
  if (flat && pool_alloc(&d_scratch, 8 * (so_at() + 2 * buckets + places), s) != RECSPLIT_OK) flat = false;
  if (!flat && pool_alloc(&d_scratch, 8 * (so_at() + 2 * buckets), s) != RECSPLIT_OK)
    return RECSPLIT_OK;  // fall back to per-query selects
  uint64_t* const d = static_cast<uint64_t*>(d_scratch);
  std::vector<uint64_t> host(base_at() + count + 1);
  uint64_t* const base = host.data() + base_at();
  uint64_t* next_so = d + so_at();
  uint64_t* keys = next_so + 2 * buckets;
  uint64_t total = 0;
  for (uint32_t i = 0; i < count; i++) {
    View& v = views[i];
    base[i] = total;
    if (v.nb) v.so = next_so;
    next_so += 2 * v.nb;
    if (flat) {
      const DecodeView dv = decode_view(*hs[i], v, keys, codes_per_part(codes));
      const FlatView f = flat_view(*hs[i], dv);
      memcpy(host.data() + i * kDecodeWords, &dv, sizeof(DecodeView));
      memcpy(host.data() + flat_at() + i * kFlatWords, &f, sizeof(FlatView));
      if (v.nb) keys += flat_places(*hs[i]);
      total += v.nb << dv.log_group;
    } else {
      memcpy(host.data() + i * kViewWords, &v, sizeof(View));
      total += v.nb;
    }
  }
  base[count] = total;
  // (a pageable copy has left the host array when cudaMemcpyAsync returns)
  cudaError_t e = cudaMemcpyAsync(d, host.data(), host.size() * sizeof(uint64_t), cudaMemcpyHostToDevice, s);
  const View* const d_views = reinterpret_cast<const View*>(d);
  if (e == cudaSuccess) {
    const uint64_t blocks = (total + 255) / 256;
    if (flat)
      k_flat_decode_views<<<static_cast<unsigned>(blocks), 256, 0, s>>>(
          reinterpret_cast<const DecodeView*>(d), d + base_at(), count, total);
    else
      k_ef_decode_views<<<static_cast<unsigned>(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(d_views, d + base_at(),
                                                                                              count, total);
    count_launch();
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    for (uint32_t i = 0; i < count; i++) views[i].so = nullptr;
    cudaFreeAsync(d_scratch, s);
    return cuda_fail(e, "decode of the structures");
  }
  *scratch = d;
  if (flat)
    batch->views = d + flat_at();
  else
    batch->decoded = d_views;
  batch->steps = steps;
  return RECSPLIT_OK;
}

View make_view(const Handle& h) {
  View v;
  v.so = nullptr;
  v.mmax = h.header[H_MMAX];
  v.extra = header_extra(h.header);
  const uint64_t* H = h.header;
  v.tree = h.d_blob + h.layout.tree;
  v.lower = h.d_blob + h.layout.lower;
  v.upper_a = h.d_blob + h.layout.upper_a;
  v.upper_b = h.d_blob + h.layout.upper_b;
  v.anchors = h.d_blob + h.layout.anchors;
  v.subs = reinterpret_cast<const uint16_t*>(h.d_blob + h.layout.subs);
  v.table = h.d_table;
  v.rec = lookup_records(h.d_table, h.table_mmax);
  v.tree_words32 = 2 * words_of_bits(H[H_TBITS]);
  v.nb = H[H_NB];
  v.beta = H[H_BETA];
  v.delta_a = static_cast<int64_t>(H[H_DELTA_A]);
  v.delta_b = static_cast<int64_t>(H[H_DELTA_B]);
  v.low_a = static_cast<uint32_t>(H[H_LOW_A]);
  v.low_b = static_cast<uint32_t>(H[H_LOW_B]);
  return v;
}

// Launch of a lookup.  `early`: the launch before it in the stream is the decode of
// the structure, whose blocks let this grid start once all of them run; it
// reads its keys and computes their signatures meanwhile and waits
// for the decode's end before it reads the decode's results (10^7 keys, l = 8,
// b = 100: 10^6 queries 37.0 -> 34.8 us).
template <typename... P, typename... A>
cudaError_t launch_lookup(bool early, void (*kernel)(P...), unsigned grid, int block, cudaStream_t s, A... args) {
  if (!early) {
    kernel<<<grid, block, 0, s>>>(P(args)...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

int lookup_structure(const Handle& h, const KeyInput& q, uint64_t* d_out, cudaStream_t s, bool allow_scratch) {
  if (q.n == 0) return RECSPLIT_OK;
  LookupRange range;
  View v = make_view(h);
  allow_scratch = allow_scratch && v.nb && q.n >= kDecodeQueries && decode_fits(h.range_size, v.mmax);
  int dev = 0, sms = 0;
  RS_CUDA(cudaGetDevice(&dev));
  RS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int block = 256;
  const uint64_t want = (q.n + block - 1) / block;
  const unsigned grid = static_cast<unsigned>(want < uint64_t(sms) * 64 ? want : uint64_t(sms) * 64);
  // With enough queries every code is decoded once (flat_pays), or else the prefix
  // sums and offsets of all buckets (decode_pays) instead of selected per query (the
  // stored structure does not change).  The scratch is allocated only then.
  const uint64_t places = allow_scratch ? flat_places(h) : 0;
  uint64_t* so = nullptr;
  if (allow_scratch && flat_pays(q.n, h.ncodes, v.nb, places) &&
      pool_alloc(reinterpret_cast<void**>(&so), 16 * v.nb + 8 * places, s) == RECSPLIT_OK) {
    View d = v;
    d.so = so;
    const DecodeView dv = decode_view(h, d, so + 2 * v.nb, codes_per_part(h.ncodes));
    const FlatView fv = flat_view(h, dv);
    const unsigned dg = static_cast<unsigned>(((v.nb << dv.log_group) + block - 1) / block);
    (v.extra ? k_flat_decode<true> : k_flat_decode<false>)<<<dg, block, 0, s>>>(dv);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
      e = q.u64 ? launch_lookup(true,
                                steps_computed(h)
                                    ? (v.extra ? k_lookup_u64_flat<true, true> : k_lookup_u64_flat<false, true>)
                                    : (v.extra ? k_lookup_u64_flat<true, false> : k_lookup_u64_flat<false, false>),
                                grid, block, s, fv, q.u64, q.n, d_out)
                : launch_lookup(true, v.extra ? k_lookup_bytes_flat<true> : k_lookup_bytes_flat<false>, grid, block, s,
                                fv, q.bytes, q.offsets, q.n, d_out);
    count_launch(2);
    cudaFreeAsync(so, s);
    if (e != cudaSuccess) return cuda_fail(e, "lookup launch");
    return RECSPLIT_OK;
  }
  if (allow_scratch && decode_pays(q.n, v.nb) &&
      pool_alloc(reinterpret_cast<void**>(&so), 16 * v.nb, s) == RECSPLIT_OK) {
    View d = v;
    d.so = so;
    const uint64_t dg = (v.nb + block - 1) / block;
    (v.extra ? k_ef_decode<true> : k_ef_decode<false>)<<<static_cast<unsigned>(dg < 65535 ? dg : 65535), block, 0,
                                                         s>>>(d);
    count_launch();
  } else {
    so = nullptr;
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = q.u64 ? launch_lookup(so != nullptr,
                              so ? (v.extra ? k_lookup_u64<true, true> : k_lookup_u64<false, true>)
                                 : (v.extra ? k_lookup_u64<true, false> : k_lookup_u64<false, false>),
                              grid, block, s, v, so, q.u64, q.n, d_out)
              : launch_lookup(so != nullptr,
                              so ? (v.extra ? k_lookup_bytes<true, true> : k_lookup_bytes<false, true>)
                                 : (v.extra ? k_lookup_bytes<true, false> : k_lookup_bytes<false, false>),
                              grid, block, s, v, so, q.bytes, q.offsets, q.n, d_out);
  count_launch();
  if (so) cudaFreeAsync(so, s);
  if (e != cudaSuccess) return cuda_fail(e, "lookup launch");
  return RECSPLIT_OK;
}

}  // namespace rs
