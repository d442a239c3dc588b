// Host-side tables: splitting strategy (Sec. 5.4), Golomb-Rice parameters
// (Sec. 5.4 Eq. gr, Sec. 7.2) and the subtree skip information of Sec. 6.2.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "common.h"

namespace rs {

Layout layout_of(const uint64_t* h) {
  Layout L;
  const uint64_t nb = h[H_NB];
  L.n_anchor = (nb >> kInvHi) + 1;
  L.n_sub = (nb >> kInvLo) + 1;
  L.tree = kHeaderWords;
  L.lower = L.tree + words_of_bits(h[H_TBITS]);
  L.upper_a = L.lower + words_of_bits((nb + 1) * (h[H_LOW_A] + h[H_LOW_B]));
  L.upper_b = L.upper_a + words_of_bits(h[H_UP_A]);
  L.anchors = L.upper_b + words_of_bits(h[H_UP_B]);
  L.subs = L.anchors + 2 * L.n_anchor;
  L.total = L.subs + (2 * L.n_sub * sizeof(uint16_t) + 7) / 8;
  return L;
}

// Sec. 5.4: s = max(2, ceil(0.35 l + 0.5)) leaves are aggregated first, then
// t = ceil(0.21 l + 0.9) (l >= 7; 2 below) such groups; the decimal
// coefficients are applied as exact fractions (7/20, 1/2, 21/100, 9/10).
Strategy make_strategy(uint32_t leaf) {
  const uint64_t l = leaf;
  uint64_t s = (7 * l + 10 + 19) / 20;
  if (s < 2) s = 2;
  const uint64_t t = l >= 7 ? (21 * l + 90 + 99) / 100 : 2;
  return Strategy{leaf, s * l, s * t * l};
}

Shape shape_of(const Strategy& st, uint64_t m) {
  if (m <= st.leaf) return Shape{0, 0, 0};
  if (m > st.upper) {
    // fanout 2; the left part is floor(m/2) rounded up to a multiple of s*t*l
    const uint64_t left = (m / 2 + st.upper - 1) / st.upper * st.upper;
    return Shape{2, left, m - left};
  }
  const uint64_t unit = m <= st.lower ? st.leaf : st.lower;
  const uint64_t fanout = (m + unit - 1) / unit;
  return Shape{static_cast<uint32_t>(fanout), unit, m - unit * (fanout - 1)};
}

static int floor_log2(uint64_t x) { return x ? 63 - __builtin_clzll(x) : 0; }

// ln k! and k ln k, each computed once per k when a whole table is built: the
// terms of the trial probabilities of all sizes are these.  (Computing both for
// every part of every size took 26 us for sizes up to 111 and 0.58 ms up to
// 2300 per class, with the device idle; once each, 8 us and 0.16 ms.)
struct LogTerms {
  std::vector<double> fact, self;
  void extend(uint64_t k) {
    for (uint64_t j = fact.size(); j <= k; j++) {
      const double dj = static_cast<double>(j);
      fact.push_back(std::lgamma(dj + 1.0));
      self.push_back(j ? dj * std::log(dj) : 0.0);
    }
  }
};

// ln of the probability that one trial succeeds at a node of m keys:
// m!/m^m for a leaf (Sec. 5.2); for a split Eq. probsplit, i.e. that times
// k^k/k! for every part k (Sec. 5.1).  With leaf range extra e a leaf trial
// succeeds when its m values are distinct in [0, R), R = m + e:
// R! / ((R - m)! R^m) (m!/m^m for e = 0).  Without terms (one size alone) the
// same values are computed in place.
static double log_trial_success(const Strategy& st, uint64_t m, const Shape& sh, LogTerms* terms) {
  auto fact = [&](uint64_t k) { return terms ? terms->fact[k] : std::lgamma(static_cast<double>(k) + 1.0); };
  auto self = [&](uint64_t k) {
    const double dk = static_cast<double>(k);
    return terms ? terms->self[k] : dk * std::log(dk);
  };
  if (sh.fanout == 0) {
    if (terms) terms->extend(m + st.extra);
    const double dm = static_cast<double>(m), dr = static_cast<double>(m + st.extra);
    return fact(m + st.extra) - fact(st.extra) - dm * std::log(dr);
  }
  if (terms) terms->extend(m);
  double v = fact(m) - self(m);
  auto term = [&](uint64_t k) { return self(k) - fact(k); };
  v += static_cast<double>(sh.fanout - 1) * term(sh.unit);
  v += term(sh.last);
  return v;
}

// lp: log_trial_success of the node
static int golomb_rice_of(uint64_t m, const Shape& sh, double lp) {
  if (m < 2) return 0;
  if (m < 65536) {
    // Eq. gr: r = max(0, ceil(lg(-lg(phi) / lg(1 - p))))
    static const double log_phi = -std::log(0.5 * (1.0 + std::sqrt(5.0)));
    const double x = std::log2(log_phi / std::log1p(-std::exp(lp)));
    const double c = std::ceil(x);
    return c > 0.0 ? static_cast<int>(c) : 0;
  }
  // Sec. 7.2 integer approximation for large nodes (">>" as a right shift)
  int64_t v = static_cast<int64_t>(((sh.fanout - 1) * 5ull) >> 1);
  v += static_cast<int64_t>(sh.fanout - 1) * floor_log2(sh.unit + (sh.unit >> 1));
  v += floor_log2(sh.last + (sh.last >> 1));
  v -= floor_log2(m);
  return v > 0 ? static_cast<int>(v >> 1) : 0;
}

int golomb_rice_param(const Strategy& st, uint64_t m) {
  if (m < 2) return 0;
  const Shape sh = shape_of(st, m);
  return golomb_rice_of(m, sh, m < 65536 ? log_trial_success(st, m, sh, nullptr) : 0.0);
}

int build_tables(uint32_t leaf, uint32_t extra, uint64_t mmax, Tables* T, std::string* err) {
  Strategy st = make_strategy(leaf);
  st.extra = extra;
  if (mmax < 2) mmax = 2;
  T->mmax = mmax;
  T->r.assign(mmax + 1, 0);
  T->fixed_bits.assign(mmax + 1, 0);
  T->codes.assign(mmax + 1, 0);
  T->expected_trials.assign(mmax + 1, 0);
  T->range.assign(mmax + 1, 0);
  T->next_max.assign(mmax + 1, 0);
  T->heaviest.assign(mmax + 1, 0.0);
  LogTerms terms;
  // the search tables, then the lookup records (two words per size)
  T->device_words.assign((kTableWords + 2) * (mmax + 1), 0);
  LookupRecord* rec = reinterpret_cast<LookupRecord*>(T->device_words.data() + kTableWords * (mmax + 1));
  // sizes 0 and 1: no code, output range m
  T->range[1] = 1;
  T->device_words[kTableWords * 1 + 3] = uint64_t(1) << 32;
  for (uint64_t m = 2; m <= mmax; m++) {
    const Shape sh = shape_of(st, m);
    const double lp = log_trial_success(st, m, sh, &terms);
    const int r = golomb_rice_of(m, sh, lp);
    T->next_max[m] = std::max(T->next_max[m - 1], std::max(sh.unit, sh.last));
    uint64_t fb = static_cast<uint64_t>(r), nc = 1;
    if (sh.fanout) {
      fb += (sh.fanout - 1) * T->fixed_bits[sh.unit] + T->fixed_bits[sh.last];
      nc += (sh.fanout - 1) * T->codes[sh.unit] + T->codes[sh.last];
    }
    T->r[m] = static_cast<uint8_t>(r);
    T->fixed_bits[m] = fb;
    T->codes[m] = nc;
    T->range[m] = sh.fanout ? (sh.fanout - 1) * T->range[sh.unit] + T->range[sh.last] : m + extra;
    // a bucket's size is read back from its output range: the range must
    // grow strictly with the size (checked for every size)
    if (T->range[m] <= T->range[m - 1] || T->range[m] >= (1ull << 32)) {
      if (err) *err = "subtree output ranges do not grow with the node size";
      return RECSPLIT_E_INVALID;
    }
    const double et = std::exp(-lp);
    T->expected_trials[m] = et > 1e18 ? ~0ull : static_cast<uint64_t>(std::ceil(et));
    T->heaviest[m] =
        std::max(T->heaviest[m - 1], sh.fanout && et >= kHeavyTrials ? et * static_cast<double>(m) : 0.0);
    if (fb >= (1ull << 32) || nc >= (1ull << 32) || r >= 32 || sh.unit >= (1ull << 32)) {
      if (err) *err = "node size too large for the device tables";
      return RECSPLIT_E_INVALID;
    }
    T->device_words[kTableWords * m] = fb | (nc << 32);
    auto heavy_flags = [&](uint64_t k) {
      const uint64_t e = T->expected_trials[k];
      uint64_t f = 0;
      for (int i = 0; i < 2; i++)
        if (k > leaf && is_heavy(e, k, kHeavyEvals[i])) f |= 1ull << i;
      return f;
    };
    uint64_t flags = heavy_flags(m);
    if (sh.fanout) flags |= heavy_flags(sh.unit) << 2 | heavy_flags(sh.last) << 4;
    T->device_words[kTableWords * m + 1] = sh.unit | (static_cast<uint64_t>(sh.fanout) << 32) |
                                           (static_cast<uint64_t>(r) << 40) | (flags << kHeavyShift);
    T->device_words[kTableWords * m + 2] = T->expected_trials[m];
    // word 3, lower half: M = ceil(2^32 / unit), with which floor(v * M / 2^32)
    // = floor(v / unit) for every v < m when (m - 1) * (M * unit - 2^32) < 2^32
    // (always for m < 2^16); 0 where that fails, and the lookup divides
    uint64_t magic = 0;
    if (sh.unit >= 2) {
      const uint64_t M = ((1ull << 32) + sh.unit - 1) / sh.unit;
      if ((m - 1) * (M * sh.unit - (1ull << 32)) < (1ull << 32)) magic = M;
    }
    T->device_words[kTableWords * m + 3] = magic | (T->range[m] << 32);
    const uint64_t unit_codes = sh.fanout ? T->codes[sh.unit] : 0;
    if (unit_codes >= (1ull << kLookupCodeBits) || sh.fanout >= 16) {
      if (err) *err = "node size too large for the lookup records";
      return RECSPLIT_E_INVALID;
    }
    rec[m].unit = static_cast<uint32_t>(sh.unit);
    rec[m].magic = static_cast<uint32_t>(magic);
    rec[m].fixed = static_cast<uint32_t>(sh.fanout ? T->fixed_bits[sh.unit] : 0);
    rec[m].info = static_cast<uint32_t>(unit_codes) | (static_cast<uint32_t>(r) << kLookupCodeBits) |
                  (sh.fanout << 28);
  }
  return RECSPLIT_OK;
}

}  // namespace rs

extern "C" int recsplit_golomb_rice_params_extra(uint32_t leaf_size, uint32_t leaf_extra, uint64_t m_hi,
                                                 uint8_t* out) {
  if (leaf_size < 1 || leaf_size > rs::kMaxLeaf || leaf_size + leaf_extra > 32 || !out) return RECSPLIT_E_INVALID;
  rs::Strategy st = rs::make_strategy(leaf_size);
  st.extra = leaf_extra;
  for (uint64_t m = 0; m <= m_hi; m++) out[m] = static_cast<uint8_t>(rs::golomb_rice_param(st, m));
  return RECSPLIT_OK;
}

extern "C" int recsplit_golomb_rice_params(uint32_t leaf_size, uint64_t m_hi, uint8_t* out) {
  if (leaf_size < 1 || leaf_size > rs::kMaxLeaf || !out) return RECSPLIT_E_INVALID;
  const rs::Strategy st = rs::make_strategy(leaf_size);
  for (uint64_t m = 0; m <= m_hi; m++) out[m] = static_cast<uint8_t>(rs::golomb_rice_param(st, m));
  return RECSPLIT_OK;
}
