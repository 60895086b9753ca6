// Descriptors of the GSUM kernel (fwd_gsum.cu): for every block of BD trials
// and group of eight channels, the distinct delay patterns and how to make
// and read their rows.
//
// Trial k of a block (first trial i0) has leaf delays d[k][j], j < 8 (channel
// 8g + j).  Its shift is e_k = d[k][0] - d[0][0] and its pattern the vector
// rel_k[j] = (d[k][j] - d[0][j]) - e_k; trials with equal patterns read one
// row at their own shifts.  Row sample u of pattern p adds leaf j at staged
// sample  (d[0][j] mod V) + rel_p[j] + u  of its span (which starts at d[0][j]
// rounded down to V samples, 16 bytes).  Every row of a (block, group) covers u
// in [0, T + e of the last trial), rounded up to whole chunks of a row maker.
//
// The sum of a group is the sum of its two halves' (leaves 0-3 and 4-7), and
// a half has few versions (relative delays of its own four leaves) in a block.
// One descriptor, in 16-byte units:
//   [0]            x = batches, y = row length
//   [1 .. BD/4]    per trial: where its first sample is, in row elements
//   then per batch of up to kGsVersions versions of the first half:
//     x = versions of the first half in it, y = of the second half that occur
//     with them; then those versions' units, the first half's first
//   A version: the staged byte offsets of its four leaves at u = 0; a second
//     half's first offset carries, from bit kGsUseBit, with which of the
//     batch's first-half versions it makes a row (rows are in that order)
#include <algorithm>
#include <future>
#include <system_error>

#include "dd_errors.h"
#include "dd_internal.h"

namespace dd {

// Keys hold a leaf's relative delay plus this, in 13 bits: at most a block's
// spread either way, which padp bounds below.
constexpr int kBias = 4096;

// The distinct values among a block's (at most 64) trials, few of them, and which
// one each trial has.  Neighbouring trials mostly have the same, so a list does:
// sorting all trials' values made a plan's descriptors take four times as long.
struct Distinct {
  uint64_t value[64];
  int of[64];
  int n = 0;
  void add(int k, uint64_t v) {  // trials in order
    uint64_t is = 0;  // (all compared: where the list is left early is hard to predict)
    for (int q = 0; q < n; ++q) is |= (uint64_t)(value[q] == v) << q;
    if (is == 0) {
      is = (uint64_t)1 << n;
      value[n++] = v;
    }
    of[k] = __builtin_ctzll(is);
  }
  void sort(int n_trials) {  // values ascending
    int from[64], to[64];
    for (int q = 0; q < n; ++q) {
      const uint64_t v = value[q];
      int at = q;
      for (; at > 0 && value[at - 1] > v; --at) value[at] = value[at - 1], from[at] = from[at - 1];
      value[at] = v;
      from[at] = q;
    }
    for (int q = 0; q < n; ++q) to[from[q]] = q;
    for (int k = 0; k < n_trials; ++k) of[k] = to[of[k]];
  }
};

// A trial's relative delays of a half group's n leaves.
static inline uint64_t half_key(const int32_t* d, const int32_t* d0, int32_t e, int n) {
  auto leaf = [&](int j) { return (uint64_t)(d[j] - d0[j] - e + kBias) << (13 * (3 - j)); };
  if (n == 4) return leaf(0) | leaf(1) | leaf(2) | leaf(3);
  uint64_t v = 0;
  for (int j = 0; j < n; ++j) v |= leaf(j);
  return v;
}

// The descriptors of pairs [f0, f1) of a trial block and a group (numbered block
// by block), every step-th of them (their index entries relative to this part's
// first unit).
static void build_pairs(const dd_plan_s& p, int bd, int T, int padp, int64_t f0, int64_t f1, int step, GsTable& t) {
  const int V = p.dtype == DD_U8_I32 ? 16 : 4;   // samples per 16 bytes
  const int es = p.dtype == DD_U8_I32 ? 1 : 4;
  const int n_g = (p.C + kGsGroup - 1) / kGsGroup;
  // A block's delays are read a cache line of channels at a time: rows of a power
  // of two channels would otherwise put all its trials' lines in one cache set.
  constexpr int kLine = 16;
  int32_t line[64][kLine];
  int32_t e[64];
  for (int64_t f = f0; f < f1; f += step) {
    const int i0 = (int)(f / n_g) * bd, g = (int)(f % n_g);
    const int c0 = g * kGsGroup, nl = std::min(kGsGroup, p.C - c0);
    const int in_line = c0 % kLine;
    if (in_line == 0 || f == f0 || step > 1)
      for (int k = 0; k < bd; ++k)
        std::copy_n(&p.delays[(size_t)std::min(i0 + k, p.n_dm - 1) * p.C + c0 - in_line],
                    std::min(kLine, p.C - c0 + in_line), line[k]);
    const int32_t* d0 = line[0] + in_line;
    // per half (leaves 0-3, 4-7): each trial's relative delays as one key,
    // 13 bits a leaf, and the distinct keys in order
    Distinct half[2];
    for (int k = 0; k < bd; ++k) {
      const int32_t* d = line[k] + in_line;
      e[k] = d[0] - d0[0];
      for (int h = 0; h < 2; ++h) half[h].add(k, half_key(d + 4 * h, d0 + 4 * h, e[k], std::min(4, nl - 4 * h)));
    }
    for (int h = 0; h < 2; ++h) half[h].sort(bd);
    // rows: the pairs of versions that occur, in the order the kernel makes
    // them (batch of first halves, then second half, then first half)
    Distinct row;
    for (int k = 0; k < bd; ++k) {
      const int first = half[0].of[k], second = half[1].of[k];
      row.add(k, (uint64_t)((first / kGsVersions * 64 + second) * 64 + first));
    }
    row.sort(bd);
    const int n_p = row.n;
    auto first_of = [&](int q) { return (int)(row.value[q] % 64); };
    auto second_of = [&](int q) { return (int)(row.value[q] / 64 % 64); };
    auto batch_of = [&](int q) { return (int)(row.value[q] / 4096); };
    // every row covers the shifts of the whole block, in whole chunks
    const int chunk = es == 1 ? kGsChunkU8 : kGsChunkF32;
    const int row_len = (T + e[bd - 1] + chunk - 1) / chunk * chunk;
    t.cap = std::max<int64_t>(t.cap, (int64_t)n_p * row_len);
    t.patterns += n_p;
    t.samples += (int64_t)n_p * row_len;
    const size_t at = t.desc.size();
    t.desc.resize(at + 1 + bd / 4);
    uint32_t* tr = reinterpret_cast<uint32_t*>(&t.desc[at + 1]);
    for (int k = 0; k < bd; ++k) tr[k] = (uint32_t)(row.of[k] * row_len + e[k]);
    auto version = [&](int h, int v) {
      uint32_t o[4];
      for (int j = 4 * h; j < 4 * h + 4; ++j) {
        // channels past the last one: the kernel keeps zeros in their spans
        const int32_t at = j < nl ? (d0[j] & (V - 1)) + (int32_t)(half[h].value[v] >> (13 * (4 * h + 3 - j)) & 0x1fff) - kBias : 0;
        o[j - 4 * h] = (uint32_t)((at + j * (T + padp)) * es);
      }
      return uint4{o[0], o[1], o[2], o[3]};
    };
    int n_batches = 0;
    for (int q = 0; q < n_p;) {
      const int bt = batch_of(q);
      const size_t head = t.desc.size();
      t.desc.push_back(uint4{});
      const int v0 = bt * kGsVersions, v1 = std::min(half[0].n, v0 + kGsVersions);
      for (int v = v0; v < v1; ++v) t.desc.push_back(version(0, v));
      int n_second = 0;
      while (q < n_p && batch_of(q) == bt) {
        const int second = second_of(q);
        uint4 rec = version(1, second);
        const size_t rat = t.desc.size();
        t.desc.push_back(rec);
        uint32_t use = 0;
        for (; q < n_p && batch_of(q) == bt && second_of(q) == second; ++q) use |= 1u << (first_of(q) - v0);
        t.desc[rat].x |= use << kGsUseBit;
        ++n_second;
      }
      t.desc[head] = uint4{(uint32_t)(v1 - v0), (uint32_t)n_second, 0, 0};
      ++n_batches;
    }
    t.desc[at] = uint4{(uint32_t)n_batches, (uint32_t)row_len, 0, 0};
    t.idx.push_back(uint2{(uint32_t)at, (uint32_t)(t.desc.size() - at)});
    t.desc_max = std::max(t.desc_max, (int)(t.desc.size() - at) * 16);
  }
}

// Staged row pitch less the tile: the block's largest spread, both ends
// rounded to V samples, and the 8 bytes a word read may take past its last
// sample; -1 where a block spans too much for the descriptors' fields.
static int pitch_pad(const dd_plan_s& p, int bd) {
  const int V = p.dtype == DD_U8_I32 ? 16 : 4;
  const int64_t pad = ((int64_t)block_spread_of(p, bd) + 2 * V + 8 + V - 1) / V * V;
  return pad > 4000 ? -1 : (int)pad;  // (keys of 13 bits, staged byte offsets below 2^24)
}

GsSample gsum_sample(const dd_plan_s& p, int bd, int T, double most) {
  const int pad = pitch_pad(p, bd);
  if (pad < 0) return {-1.0, 0.0};
  GsTable t;
  // (whole blocks: a last one of few trials has few patterns but takes as long)
  const int n_b = std::max(1, p.n_dm / bd), n_g = (p.C + kGsGroup - 1) / kGsGroup;
  auto average = [&](int64_t sum) { return (double)sum / (double)t.idx.size(); };
  for (int k = 0; k < 4; ++k) {
    const int64_t b = (int64_t)k * n_b / 4;
    build_pairs(p, bd, T, pad, b * n_g, (b + 1) * n_g, std::max(1, n_g / 16), t);
    if (average(t.patterns) > 2.0 * most) break;  // far too many
  }
  return {average(t.patterns), average(t.samples)};
}

void gsum_build(const dd_plan_s& p, std::vector<GsTable>& tables) {
  for (GsTable& t : tables) t.padp = pitch_pad(p, t.bd);
  // the pairs are independent: up to eight threads make equal shares of every
  // table's (starting threads takes longer than a small table)
  constexpr int kParts = 8;
  std::vector<GsTable> part(tables.size() * kParts);
  auto make = [&](int k) {
    for (size_t j = 0; j < tables.size(); ++j) {
      const GsTable& t = tables[j];
      const int64_t n = (int64_t)((p.n_dm + t.bd - 1) / t.bd) * ((p.C + kGsGroup - 1) / kGsGroup);
      if (t.padp >= 0)
        build_pairs(p, t.bd, t.T, t.padp, n * k / kParts, n * (k + 1) / kParts, 1, part[j * kParts + k]);
    }
  };
  std::vector<std::future<void>> others;
  for (int k = 1; k < kParts; ++k) {
    try {
      others.push_back(std::async(std::launch::async, make, k));
    } catch (const std::system_error&) {  // no thread to be had
      make(k);
    }
  }
  make(0);
  for (auto& o : others) o.get();
  for (size_t j = 0; j < tables.size(); ++j) {
    GsTable& t = tables[j];
    for (int k = 0; k < kParts; ++k) {
      const GsTable& q = part[j * kParts + k];
      const uint32_t at = (uint32_t)t.desc.size();
      for (uint2 e : q.idx) t.idx.push_back(uint2{e.x + at, e.y});
      t.desc.insert(t.desc.end(), q.desc.begin(), q.desc.end());
      t.desc_max = std::max(t.desc_max, q.desc_max);
      t.cap = std::max(t.cap, q.cap);
    }
    // what a leaf read past the end of the last span may touch (the reads of
    // samples no row uses) stays inside the rows
    t.cap = std::max<int64_t>(t.cap, t.padp + 512);
    t.cap = (t.cap + 16 + 63) / 64 * 64;
    t.fits = t.padp >= 0 && t.cap <= 1 << 20 && t.desc.size() < (size_t)1 << 31;
  }
}

}  // namespace dd
