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
//   [0]            x = batches, y = row length, z = rows
//   [1 .. BD/4]    per trial: where its first sample is, in row elements
//   then per batch of up to kGsVersions versions of the first half:
//     x = versions of the first half in it, y = of the second half that occur
//     with them; then those versions' units, the first half's first
//   A version: the staged byte offsets of its four leaves at u = 0; a second
//     half's first offset carries, from bit kGsUseBit, with which of the
//     batch's first-half versions it makes a row (rows are in that order)
#include <algorithm>
#include <cstring>
#include <future>
#include <system_error>

#include "dd_errors.h"
#include "dd_internal.h"

namespace dd {

// Keys hold a leaf's relative delay plus this, in 13 bits: at most a block's
// spread either way, which padp bounds below.
constexpr int kBias = 4096;

// The descriptors of trial blocks [b0, b1) and every step-th group (their
// index entries relative to this part's first unit).
static void build_blocks(const dd_plan_s& p, int bd, int T, int padp, int b0, int b1, int step, GsTable& t) {
  const int V = p.dtype == DD_U8_I32 ? 16 : 4;   // samples per 16 bytes
  const int es = p.dtype == DD_U8_I32 ? 1 : 4;
  const int n_g = (p.C + kGsGroup - 1) / kGsGroup;
  uint64_t key[2][64];
  int32_t e[64];
  for (int b = b0; b < b1; ++b) {
    const int i0 = b * bd;
    for (int g = 0; g < n_g; g += step) {
      const int c0 = g * kGsGroup, nl = std::min(kGsGroup, p.C - c0);
      const int32_t* d0 = &p.delays[(size_t)i0 * p.C + c0];
      // per half (leaves 0-3, 4-7): each trial's relative delays as one key,
      // 13 bits a leaf, and the distinct keys in order
      uint64_t ver[2][64];
      int n_v[2], of[2][64];
      for (int k = 0; k < bd; ++k) {
        const int32_t* d = &p.delays[(size_t)std::min(i0 + k, p.n_dm - 1) * p.C + c0];
        e[k] = d[0] - d0[0];
        for (int h = 0; h < 2; ++h) {
          uint64_t v = 0;
          for (int j = 4 * h; j < std::min(nl, 4 * h + 4); ++j)
            v |= (uint64_t)(d[j] - d0[j] - e[k] + kBias) << (13 * (4 * h + 3 - j));
          key[h][k] = v;
        }
      }
      for (int h = 0; h < 2; ++h) {
        std::copy(key[h], key[h] + bd, ver[h]);
        std::sort(ver[h], ver[h] + bd);
        n_v[h] = (int)(std::unique(ver[h], ver[h] + bd) - ver[h]);
        for (int k = 0; k < bd; ++k) of[h][k] = (int)(std::lower_bound(ver[h], ver[h] + n_v[h], key[h][k]) - ver[h]);
      }
      // rows: the pairs of versions that occur, in the order the kernel makes
      // them (batch of first halves, then second half, then first half)
      int order[64], n_p = 0;
      auto rank = [&](int k) { return (of[0][k] / kGsVersions * 64 + of[1][k]) * 64 + of[0][k]; };
      int by[64];
      for (int k = 0; k < bd; ++k) by[k] = k;
      std::stable_sort(by, by + bd, [&](int x, int y) { return rank(x) < rank(y); });
      for (int s = 0; s < bd; ++s) {
        const int k = by[s];
        if (s == 0 || rank(k) != rank(by[s - 1])) order[n_p++] = k;
      }
      // every row covers the shifts of the whole block, in whole chunks
      const int chunk = es == 1 ? kGsChunkU8 : kGsChunkF32;
      const int row_len = (T + e[bd - 1] + chunk - 1) / chunk * chunk;
      t.cap = std::max<int64_t>(t.cap, (int64_t)n_p * row_len);
      t.patterns += n_p;
      t.samples += (int64_t)n_p * row_len;
      const size_t at = t.desc.size();
      t.desc.resize(at + 1 + bd / 4);
      uint32_t* tr = reinterpret_cast<uint32_t*>(&t.desc[at + 1]);
      for (int s = 0, q = -1; s < bd; ++s) {
        const int k = by[s];
        if (s == 0 || rank(k) != rank(by[s - 1])) ++q;
        tr[k] = (uint32_t)(q * row_len + e[k]);
      }
      auto version = [&](int h, int v) {
        uint32_t o[4];
        for (int j = 4 * h; j < 4 * h + 4; ++j) {
          // channels past the last one: the kernel keeps zeros in their spans
          const int32_t at = j < nl ? (d0[j] & (V - 1)) + (int32_t)(ver[h][v] >> (13 * (4 * h + 3 - j)) & 0x1fff) - kBias : 0;
          o[j - 4 * h] = (uint32_t)((at + j * (T + padp)) * es);
        }
        return uint4{o[0], o[1], o[2], o[3]};
      };
      int n_batches = 0;
      for (int q = 0; q < n_p;) {
        const int bt = of[0][order[q]] / kGsVersions;
        const size_t head = t.desc.size();
        t.desc.push_back(uint4{});
        const int v0 = bt * kGsVersions, v1 = std::min(n_v[0], v0 + kGsVersions);
        for (int v = v0; v < v1; ++v) t.desc.push_back(version(0, v));
        int n_second = 0;
        while (q < n_p && of[0][order[q]] / kGsVersions == bt) {
          const int second = of[1][order[q]];
          uint4 rec = version(1, second);
          const size_t rat = t.desc.size();
          t.desc.push_back(rec);
          uint32_t use = 0;
          for (; q < n_p && of[0][order[q]] / kGsVersions == bt && of[1][order[q]] == second; ++q)
            use |= 1u << (of[0][order[q]] - v0);
          t.desc[rat].x |= use << kGsUseBit;
          ++n_second;
        }
        t.desc[head] = uint4{(uint32_t)(v1 - v0), (uint32_t)n_second, 0, 0};
        ++n_batches;
      }
      t.desc[at] = uint4{(uint32_t)n_batches, (uint32_t)row_len, (uint32_t)n_p, 0};
      t.idx.push_back(uint2{(uint32_t)at, (uint32_t)(t.desc.size() - at)});
      t.desc_max = std::max(t.desc_max, (int)(t.desc.size() - at) * 16);
    }
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

GsSample gsum_sample(const dd_plan_s& p, int bd, int T) {
  const int pad = pitch_pad(p, bd);
  if (pad < 0) return {-1.0, 0.0};
  GsTable t;
  // (whole blocks: a last one of few trials has few patterns but takes as long)
  const int n_b = std::max(1, p.n_dm / bd), n_g = (p.C + kGsGroup - 1) / kGsGroup;
  for (int k = 0; k < 4; ++k) {
    const int b = (int)((int64_t)k * n_b / 4);
    build_blocks(p, bd, T, pad, b, b + 1, std::max(1, n_g / 16), t);
  }
  return {(double)t.patterns / (double)t.idx.size(), (double)t.samples / (double)t.idx.size()};
}

bool gsum_build(const dd_plan_s& p, int bd, int T, GsTable& t) {
  t = GsTable{};
  t.padp = pitch_pad(p, bd);
  if (t.padp < 0) return false;
  // trial blocks are independent: up to eight threads make equal shares
  const int n_b = (p.n_dm + bd - 1) / bd;
  const int n_parts = std::min(8, n_b);
  std::vector<GsTable> part(n_parts);
  auto make = [&](int k) {
    build_blocks(p, bd, T, t.padp, (int)((int64_t)n_b * k / n_parts), (int)((int64_t)n_b * (k + 1) / n_parts), 1,
                 part[k]);
  };
  std::vector<std::future<void>> others;
  for (int k = 1; k < n_parts; ++k) {
    try {
      others.push_back(std::async(std::launch::async, make, k));
    } catch (const std::system_error&) {  // no thread to be had
      make(k);
    }
  }
  make(0);
  for (auto& o : others) o.get();
  for (const GsTable& q : part) {
    const uint32_t at = (uint32_t)t.desc.size();
    for (uint2 e : q.idx) t.idx.push_back(uint2{e.x + at, e.y});
    t.desc.insert(t.desc.end(), q.desc.begin(), q.desc.end());
    t.desc_max = std::max(t.desc_max, q.desc_max);
    t.patterns += q.patterns;
    t.cap = std::max(t.cap, q.cap);
  }
  // what a leaf read past the end of the last span may touch (the reads of
  // samples no row uses) stays inside the rows
  t.cap = std::max<int64_t>(t.cap, t.padp + 512);
  t.cap = (t.cap + 16 + 63) / 64 * 64;
  return t.cap <= 1 << 20 && t.desc.size() < (size_t)1 << 31;
}

}  // namespace dd
