// GSUM forward kernel: sums of eight adjacent channels, made once per delay
// pattern in shared memory and used by every DM trial of the block that has it.
//
// Section 2 notes that nearby DM trials read nearly the same input samples.
// More than the samples can be shared: between neighbouring trials the delays
// of eight adjacent channels nearly always move together, so their sum
//   S_p[u] = sum_{j < 8} in[8g + j][t0 + u + (leaf j's delay in pattern p)]
// is the same series for all trials with the same relative delays (the
// pattern p), read at the trial's own shift e_i:
//   out[i][t0 + t] = sum_g S_{p(i, g)}[t + e_i].
// On the Apertif grid a block of 32 trials has 8.7 patterns per eight
// channels on average, so a trial costs one shared-memory read per eight
// channels and sample and its share of the patterns 0.10 more per channel,
// where a kernel that shares only samples (STAGED) reads eight.
//
// The sum of eight is the sum of two halves', and a half has still fewer
// versions (4 to 5 a block of 64 trials), so a row costs one add and one store.
//
//  * A block owns BD = NC * DPW trials x T = 32 * SPL samples; a summing thread
//    keeps DPW x SPL sums in registers.
//  * One warp copies: per group of eight channels the channels' spans and the
//    group's descriptor (gsum_plan.cpp), SS groups ahead.
//  * NS sets of NP warps make rows, the sets taking groups in turn: a warp makes
//    128 samples (uint8: 256) of every row of its group from the descriptor's
//    versions.
//  * NC warps add: one shared-memory read per trial, sample and group.
// Rings of mbarriers join them (RB groups of rows); nothing in the group loop
// is block-wide.
//
// What bounds it is shared memory (57 % of its cycles on uint8, 68 on float) and the
// chain of its reads in the row makers.  One Apertif uint8 beam (1024 x 2048 x
// 20,000; u8pk takes 2.09 ms), each step measured: every warp making rows and
// adding between two block barriers 3.7 ms (one warp's chain of dependent reads
// holds all up), row makers apart 2.5, leaves all read for every version
// instead of the changed ones behind predicates 2.4 (a predicated-off read
// still takes its turn), rings and two sets 1.8, three sets 1.5, spans two
// rounds of the sets ahead (a set otherwise waits out its own copy) 1.43, two
// words a lane and tiles of 576 samples (448: 1.39 ms with four sets) 1.39.
// Eight versions kept instead of six: 1.55; waits that suspend the warp: 1.47.
//
// Float sums are (x0 + x1 + x2 + x3) + (x4 + x5 + x6 + x7) within eight
// channels, then one add to the running sum, in channel order.  8-bit sums are
// exact: rows hold 16-bit sums (at most 8 * 255), two per word; the packed sums
// are added for 32 groups (32 * 8 * 255 < 65536) and then added to the output.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dd_internal.h"
#include "ptx.cuh"

namespace dd {

namespace {

constexpr int kG = kGsGroup;
constexpr int kHeadBytes = 512;
constexpr int kMaxRing = 6;

struct GsHead {
  uint64_t sfull[kMaxRing];   // a group's spans and descriptor have landed
  uint64_t sempty[kMaxRing];  // the row makers are done with them
  uint64_t rfull[kMaxRing];   // a group's rows are made
  uint64_t rempty[kMaxRing];  // the summing warps are done with them
};
static_assert(sizeof(GsHead) <= kHeadBytes, "header");

// The 4 bytes starting at byte (sel mod 4) of the 8 bytes lo, hi (lo first).
__device__ __forceinline__ uint32_t bytes_from(uint32_t lo, uint32_t hi, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32.f4e %0, %1, %2, %3;" : "=r"(d) : "r"(lo), "r"(hi), "r"(sel));
  return d;
}

// ------------------------------------------------------- rows, float
__device__ __forceinline__ void sum2_rn(float& r0, float& r1, float a0, float a1, float b0, float b1) {
  asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 x, x, y;\n"
      " mov.b64 {%0, %1}, x;\n}\n"
      : "=f"(r0), "=f"(r1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// The rows of one group over the samples [u0, u0 + 128): lane l makes u0 + l + 32 q.
struct RowMaker {
  static constexpr int kKeep = kGsVersions;
  const FwdArgs& a;
  const GsLaunch& gs;
  const char* src;  // sample u0 + lane of the stage
  float* dst;       // where the next row's sample u0 + lane goes
  const float* end;
  int u0, row_len;
  using Sum = float[4];

  __device__ __forceinline__ RowMaker(const FwdArgs& a_, const GsLaunch& gs_, const float* st, float* rows, int row_len_,
                                      int u0_, int lane)
      : a(a_), gs(gs_), src(reinterpret_cast<const char*>(st + u0_ + lane)), dst(rows + u0_ + lane),
        end(rows + gs_.cap), u0(u0_), row_len(row_len_) {}
  // the sum of a version's four leaves
  __device__ __forceinline__ void sum(const uint4& v, Sum& t) {
    uint32_t o[4] = {v.x, v.y, v.z, v.w};
    float leaf[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!DD_INDEX_OK(a.status, (int)o[j] / 4 + u0 + 128 <= gs.reach)) o[j] = 0;
      const float* s = reinterpret_cast<const float*>(src + o[j]);
#pragma unroll
      for (int q = 0; q < 4; ++q) leaf[j][q] = s[32 * q];
    }
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      sum2_rn(t[q], t[q + 1], leaf[0][q], leaf[0][q + 1], leaf[1][q], leaf[1][q + 1]);
      add2_rn(t[q], t[q + 1], leaf[2][q], leaf[2][q + 1]);
      add2_rn(t[q], t[q + 1], leaf[3][q], leaf[3][q + 1]);
    }
  }
  __device__ __forceinline__ void store(const Sum& x, const Sum& y) {
    float t[4];
#pragma unroll
    for (int q = 0; q < 4; q += 2) sum2_rn(t[q], t[q + 1], x[q], x[q + 1], y[q], y[q + 1]);
    if (DD_INDEX_OK(a.status, dst + 96 < end)) {
#pragma unroll
      for (int q = 0; q < 4; ++q) dst[32 * q] = t[q];
    }
    dst += row_len;
  }
};

// ------------------------------------------------------- rows, uint8
// Lane l makes the four samples from u = u0 + 4 l on, and the four 128 further.  A leaf is one word,
// taken from the two aligned words around it; four leaves' words added mod
// 2^32 give A, their odd bytes in two 16-bit lanes O = S1 + 2^16 S3, and A -
// 2^8 O = S0 + 2^16 S2.
struct RowMakerU8 {
  static constexpr int kKeep = kGsVersions;
  static constexpr int kWords = kGsChunkU8 / 128;  // a lane's words, 128 samples apart
  const FwdArgs& a;
  const GsLaunch& gs;
  const uint8_t* src;  // sample u of the stage (u, T and the stage are multiples of 4)
  uint16_t* dst;
  const uint16_t* end;
  int u, row_len;
  using Sum = uint32_t[2 * kWords];  // of each word S0 + 2^16 S2, S1 + 2^16 S3

  __device__ __forceinline__ RowMakerU8(const FwdArgs& a_, const GsLaunch& gs_, const uint8_t* st, uint16_t* rows,
                                        int row_len_, int u0, int lane)
      : a(a_), gs(gs_), src(st + u0 + 4 * lane), dst(rows + u0 + 4 * lane), end(rows + gs_.cap), u(u0 + 4 * lane),
        row_len(row_len_) {}
  __device__ __forceinline__ void sum(const uint4& v, Sum& t) {
    uint32_t o[4] = {v.x, v.y, v.z, v.w};
    uint32_t A[kWords], O[kWords];
#pragma unroll
    for (int q = 0; q < kWords; ++q) A[q] = O[q] = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!DD_INDEX_OK(a.status, (int)o[j] + u + 128 * kWords - 120 <= gs.reach)) o[j] = 0;
      const uint32_t* s = reinterpret_cast<const uint32_t*>(src + (o[j] & ~3u));
#pragma unroll
      for (int q = 0; q < kWords; ++q) {
        const uint32_t x = bytes_from(s[32 * q], s[32 * q + 1], o[j]);
        A[q] += x;
        O[q] += __byte_perm(x, 0u, 0x4341u);
      }
    }
#pragma unroll
    for (int q = 0; q < kWords; ++q) {
      t[2 * q] = A[q] - (O[q] << 8);
      t[2 * q + 1] = O[q];
    }
  }
  __device__ __forceinline__ void store(const Sum& x, const Sum& y) {
    if (DD_INDEX_OK(a.status, dst + 128 * kWords - 124 <= end)) {
#pragma unroll
      for (int q = 0; q < kWords; ++q) {
        const uint32_t E = x[2 * q] + y[2 * q], O = x[2 * q + 1] + y[2 * q + 1];
        *reinterpret_cast<uint2*>(dst + 128 * q) = make_uint2(__byte_perm(E, O, 0x5410u), __byte_perm(E, O, 0x7632u));
      }
    }
    dst += row_len;
  }
};

// One warp, one chunk of samples of a group's rows: the versions of the first half's
// sum stay in registers, kKeep at a time; each version of the second
// half's sum is made once per such batch and added to those it occurs with.
template <typename Maker>
__device__ __forceinline__ void make_rows(Maker& mk, const uint4* d, int n_batches) {
#pragma unroll 1
  for (int bt = 0; bt < n_batches; ++bt) {
    const uint4 h = *d++;  // x = versions of the first half, y = of the second half
    typename Maker::Sum A[Maker::kKeep];
#pragma unroll
    for (int v = 0; v < Maker::kKeep; ++v)
      if (v < (int)h.x) mk.sum(d[v], A[v]);
    d += h.x;
    uint4 rec = *d++;
#pragma unroll 1
    for (int k = (int)h.y; k > 0; --k) {
      const uint32_t use = rec.x >> kGsUseBit;
      rec.x &= kGsOffsetMask;
      typename Maker::Sum Bv;
      mk.sum(rec, Bv);
      if (k > 1) rec = *d++;
#pragma unroll
      for (int v = 0; v < Maker::kKeep; ++v)
        if (use & (1u << v)) mk.store(A[v], Bv);
    }
  }
}

template <typename Tin>
struct GsTypes;
template <>
struct GsTypes<float> {
  using Row = float;
  using Out = float;
  using Maker = RowMaker;
};
template <>
struct GsTypes<uint8_t> {
  using Row = uint16_t;
  using Out = int32_t;
  using Maker = RowMakerU8;
};

// ------------------------------------------------------- stage 2: the sums
template <typename Tin, int DPW, int SPL>
struct Sums;

template <int DPW, int SPL>
struct Sums<float, DPW, SPL> {
  static_assert(SPL % 2 == 0, "packed pairs");
  float acc[DPW][SPL];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int m = 0; m < DPW; ++m)
#pragma unroll
      for (int q = 0; q < SPL; ++q) acc[m][q] = 0.0f;
  }
  __device__ __forceinline__ void add(const float* rows, const uint32_t (&off)[DPW], int lane) {
#pragma unroll
    for (int m = 0; m < DPW; ++m) {
      const float* r = rows + off[m] + lane;
#pragma unroll
      for (int q = 0; q < SPL; q += 2) add2_rn(acc[m][q], acc[m][q + 1], r[32 * q], r[32 * q + 32]);
    }
  }
  __device__ __forceinline__ void flush(const FwdArgs& a, float*, int i, int64_t t0, int lane, bool) {
    float* __restrict__ out = static_cast<float*>(a.out);
#pragma unroll
    for (int m = 0; m < DPW; ++m) {
      if (i + m >= a.n_dm) break;
      float* o = out + (int64_t)(i + m) * a.out_stride + t0 + lane;
#pragma unroll
      for (int q = 0; q < SPL; ++q)
        if (t0 + lane + 32 * q < a.n_out) o[32 * q] = acc[m][q];
    }
  }
};

// A lane owns SPL consecutive samples: KW = SPL / 2 words of two 16-bit sums
// (KW odd: the lanes' word reads hit distinct banks).
template <int DPW, int SPL>
struct Sums<uint8_t, DPW, SPL> {
  static constexpr int KW = SPL / 2;
  static_assert(SPL % 4 == 2, "an odd number of words per lane");
  uint32_t pk[DPW][KW];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int m = 0; m < DPW; ++m)
#pragma unroll
      for (int q = 0; q < KW; ++q) pk[m][q] = 0u;
  }
  __device__ __forceinline__ void add(const uint16_t* rows, const uint32_t (&off)[DPW], int lane) {
#pragma unroll
    for (int m = 0; m < DPW; ++m) {
      const uint32_t* r = reinterpret_cast<const uint32_t*>(rows) + (off[m] >> 1) + KW * lane;
      const uint32_t sel = 2u * (off[m] & 1u);  // an odd start takes its samples across two words
      uint32_t lo = r[0];
#pragma unroll
      for (int q = 0; q < KW; ++q) {
        const uint32_t hi = r[q + 1];
        pk[m][q] += bytes_from(lo, hi, sel);
        lo = hi;
      }
    }
  }
  // Add the packed sums to the output (the first time: store them) and clear
  // them; the samples turn through the warp's own part of shared memory, so
  // that lanes run along time.
  __device__ __forceinline__ void flush(const FwdArgs& a, int32_t* turn, int i, int64_t t0, int lane, bool first) {
    int32_t* __restrict__ out = static_cast<int32_t*>(a.out);
#pragma unroll
    for (int m = 0; m < DPW; ++m) {
      if (i + m < a.n_dm) {
#pragma unroll
        for (int q = 0; q < KW; ++q) {
          turn[lane * SPL + 2 * q] = (int32_t)(pk[m][q] & 0xffffu);
          turn[lane * SPL + 2 * q + 1] = (int32_t)(pk[m][q] >> 16);
        }
        __syncwarp();
        int32_t* o = out + (int64_t)(i + m) * a.out_stride + t0 + lane;
        int32_t v[SPL];
#pragma unroll
        for (int q = 0; q < SPL; ++q) v[q] = !first && t0 + lane + 32 * q < a.n_out ? o[32 * q] : 0;
#pragma unroll
        for (int q = 0; q < SPL; ++q)
          if (t0 + lane + 32 * q < a.n_out) o[32 * q] = v[q] + turn[lane + 32 * q];
        __syncwarp();
      }
#pragma unroll
      for (int q = 0; q < KW; ++q) pk[m][q] = 0u;
    }
  }
};

// Three kinds of warps, each running ahead of the next as far as its ring
// lets it: one copies spans (SS groups), NS sets of NP warps make rows (RB
// groups; the sets take groups in turn, as the chain of reads that makes one
// group's rows takes longer than adding them), NC add them up.  Every wait is
// bounded; a warp whose wait ran out goes through its remaining groups
// without waiting or working and stores nothing more.  It reports the timeout;
// what the launch's output holds then is undefined (other warps store theirs).
template <typename Tin, int NC, int NS, int NP, int DPW, int SPL, int SS, int RB, int MB>
__global__ void __launch_bounds__(32 * (NC + NS * NP + 1), MB) fwd_gsum_kernel(FwdArgs a, GsLaunch gs) {
  using Row = typename GsTypes<Tin>::Row;
  constexpr int V = 16 / (int)sizeof(Tin);
  constexpr int BD = NC * DPW, T = 32 * SPL;
  static_assert(kDmPad % BD == 0, "a block's trials stay inside the padded delay row");
  static_assert(T % V == 0 && (DPW == 1 || DPW == 2 || DPW % 4 == 0), "tile shape");
  // A parity wait tells a phase only from the next: the wait for a ring
  // entry's n-th completion needs the (n - 1)-th to be over.  The spans of
  // group g - SS were waited for by the same set if SS is a multiple of NS;
  // rows g - NS could be made only when g - NS - RB, hence g - 2 RB, was added.
  static_assert(SS <= kMaxRing && RB <= kMaxRing && SS % NS == 0 && NS <= RB, "rings");
  extern __shared__ __align__(128) unsigned char smem[];
  GsHead& B = *reinterpret_cast<GsHead*>(smem);
  uint32_t* const offs = reinterpret_cast<uint32_t*>(smem + kHeadBytes);  // [RB][BD]: where each trial's samples start
  unsigned char* const dring = smem + kHeadBytes + RB * BD * 4;           // [SS] descriptors
  const int pitch = T + gs.padp;
  const int stage_bytes = kG * pitch * (int)sizeof(Tin);
  unsigned char* const sring = dring + SS * gs.desc_max;                   // [SS] spans
  Row* const rows = reinterpret_cast<Row*>(sring + SS * stage_bytes);      // [RB][cap]
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int b = blockIdx.x, i0 = b * BD;
  const int64_t t0 = (int64_t)blockIdx.y * T;
  const int ng = (a.C + kG - 1) / kG;

  if (tid == 0) {
    for (int k = 0; k < SS; ++k) mbar_init(&B.sfull[k], 1), mbar_init(&B.sempty[k], NP);
    for (int k = 0; k < RB; ++k) mbar_init(&B.rfull[k], NP), mbar_init(&B.rempty[k], NC);
    fence_mbar_init();
  }
  __syncthreads();
  bool ok = true;
  // wait until ring entry g % N of `bar` has completed for the (g / N)-th time (bounded, warp-uniform)
  auto wait = [&](uint64_t* bar, int n) {
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar, (uint32_t)(n & 1), kWaitLimitCycles));
  };

  if (warp == NC + NS * NP) {
    // Copies: lane j < 8 channel 8g + j's span, lane 8 the descriptor; what a
    // copy needs from memory is read one group before (fetch).
    const int nt = (int)min((int64_t)T, a.n_out - t0);
    int f0 = 0, f1 = 0;
    auto fetch = [&](int g) {
      if (g >= ng) return;
      if (lane < kG) {
        const int c = kG * g + lane;
        if (c < a.C) {
          const int32_t* col = a.delaysT + (int64_t)c * a.n_dm_pad + i0;
          f0 = __ldg(col);
          f1 = __ldg(col + BD - 1);
        }
      } else if (lane == kG) {
        const uint2 e = __ldg(gs.idx + (int64_t)b * ng + g);
        f0 = (int)e.x, f1 = (int)e.y;
      }
    };
    fetch(0);
    int g = 0;
    for (; g < ng; ++g) {
      const int k = g % SS;
      if (g >= SS) wait(&B.sempty[k], g / SS - 1);
      if (!ok) break;
      const int c = kG * g + lane;
      const bool span = lane < kG && c < a.C;
      int64_t al = 0, ah = 0;
      if (span) {
        al = (t0 + f0) & ~(int64_t)(V - 1);
        ah = (t0 + nt + f1 + V - 1) & ~(int64_t)(V - 1);
        if (!DD_INDEX_OK(a.status, al >= 0 && ah - al <= pitch && ah <= a.in_avail)) al = 0, ah = V;
      }
      unsigned char* st = sring + k * stage_bytes;
      // channels past the last one count as zeros
      for (int j = a.C - kG * g; j < kG; ++j) {
        uint4* z = reinterpret_cast<uint4*>(st + j * pitch * (int)sizeof(Tin));
        for (int m = lane; m < pitch / V; m += 32) z[m] = uint4{0, 0, 0, 0};
      }
      const uint32_t bytes = span ? (uint32_t)((ah - al) * (int64_t)sizeof(Tin)) : lane == kG ? (uint32_t)f1 * 16u : 0u;
      const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
      __syncwarp();
      if (lane == 0) mbar_arrive_expect_tx(&B.sfull[k], total);
      __syncwarp();
      if (span)
        bulk_g2s(st + lane * pitch * (int)sizeof(Tin), static_cast<const Tin*>(a.in) + (int64_t)c * a.in_stride + al,
                 bytes, &B.sfull[k]);
      else if (lane == kG)
        bulk_g2s(dring + k * gs.desc_max, gs.desc + f0, bytes, &B.sfull[k]);
      fetch(g + 1);
    }
    // no copy may be in flight when the block leaves
    for (int m = max(0, g - SS); m < g; ++m)
      (void)mbar_wait_bounded(&B.sfull[m % SS], (uint32_t)(m / SS & 1), kWaitLimitCycles);
    if (!ok && lane == 0) report_error(a.status, kDevWaitTimeout);
    return;
  }

  if (warp >= NC) {
    constexpr int kChunk = sizeof(Tin) == 1 ? kGsChunkU8 : kGsChunkF32;
    const int set = (warp - NC) / NP, pw = (warp - NC) % NP;
    for (int g = set; g < ng; g += NS) {
      const int k = g % SS, r = g % RB;
      wait(&B.sfull[k], g / SS);
      if (g >= RB) wait(&B.rempty[r], g / RB - 1);
      if (ok) {
        const uint4* d = reinterpret_cast<const uint4*>(dring + k * gs.desc_max);
        const uint4 h = d[0];
        if (pw == NP - 1)
          for (int m = lane; m < BD; m += 32) offs[r * BD + m] = reinterpret_cast<const uint32_t*>(d + 1)[m];
        for (int u0 = kChunk * pw; u0 < (int)h.y; u0 += kChunk * NP) {
          typename GsTypes<Tin>::Maker mk(a, gs, reinterpret_cast<const Tin*>(sring + k * stage_bytes),
                                          rows + r * gs.cap, (int)h.y, u0, lane);
          make_rows(mk, d + 1 + BD / 4, (int)h.x);
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&B.rfull[r]);
        mbar_arrive(&B.sempty[k]);
      }
    }
    if (!ok && lane == 0) report_error(a.status, kDevWaitTimeout);
    return;
  }

  Sums<Tin, DPW, SPL> s;
  s.clear();
  typename GsTypes<Tin>::Out* turn =
      reinterpret_cast<typename GsTypes<Tin>::Out*>(rows + (size_t)RB * gs.cap) + warp * T;
  bool first = true;
  for (int g = 0; g < ng; ++g) {
    const int r = g % RB;
    wait(&B.rfull[r], g / RB);
    if (ok) {
      const uint32_t* tr = offs + r * BD + warp * DPW;
      uint32_t off[DPW];
      if constexpr (DPW % 4 == 0) {
#pragma unroll
        for (int m = 0; m < DPW; m += 4) {
          const uint4 v = *reinterpret_cast<const uint4*>(tr + m);
          off[m] = v.x, off[m + 1] = v.y, off[m + 2] = v.z, off[m + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int m = 0; m < DPW; ++m) off[m] = tr[m];
      }
#pragma unroll
      for (int m = 0; m < DPW; ++m)
        if (!DD_INDEX_OK(a.status, off[m] + T <= (uint32_t)gs.cap)) off[m] = 0;
      s.add(rows + r * gs.cap, off, lane);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&B.rempty[r]);
    // 16-bit sums hold 32 groups
    if (sizeof(Tin) == 1 && (g & 31) == 31 && g + 1 < ng && ok) {
      s.flush(a, turn, i0 + warp * DPW, t0, lane, first);
      first = false;
    }
  }
  if (ok)
    s.flush(a, turn, i0 + warp * DPW, t0, lane, first);
  else if (lane == 0)
    report_error(a.status, kDevWaitTimeout);
}

// X(type, summing warps, row-making sets, warps each, trials per summing warp,
//   samples per lane, span ring, row ring, blocks per SM)
#define DD_GSUM_F32(X)                 \
  X(float, 16, 2, 5, 4, 12, 2, 2, 1)
#define DD_GSUM_U8(X)                  \
  X(uint8_t, 16, 3, 3, 4, 18, 6, 3, 1) \
  X(uint8_t, 16, 4, 3, 4, 14, 4, 4, 1) \
  X(uint8_t, 8, 3, 3, 4, 14, 6, 4, 1)  \
  X(uint8_t, 8, 2, 2, 2, 14, 4, 3, 2)

#define GS_P NC, NS, NP, DPW, SPL, SS, RB, MB
template <typename Tin, int NC, int NS, int NP, int DPW, int SPL, int SS, int RB, int MB>
cudaError_t launch_t(const TileConfig& cfg, const FwdArgs& a, cudaStream_t s) {
  auto kern = fwd_gsum_kernel<Tin, GS_P>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, cfg.smem);
  if (e != cudaSuccess) return e;
  constexpr int BD = NC * DPW, T = 32 * SPL;
  dim3 grid((unsigned)((a.n_dm + BD - 1) / BD), (unsigned)((a.n_out + T - 1) / T));
  if (grid.y > 65535) return cudaErrorInvalidConfiguration;
  kern<<<grid, 32 * (NC + NS * NP + 1), cfg.smem, s>>>(a, cfg.gs);
  return cudaGetLastError();
}

}  // namespace

#define GS_IS(NC, NS, NP, DPW, SPL, SS, RB, MB)                                                     \
  (cfg.threads == 32 * (NC + NS * NP + 1) && cfg.bd == NC * DPW && cfg.bt == 32 * SPL && cfg.stages == SS && \
   cfg.cc == RB)
cudaError_t launch_gsum(const TileConfig& cfg, dd_dtype dtype, const FwdArgs& a, cudaStream_t s) {
  // no weights (float plans that have GSUM are the adjoint's, which scales its
  // result), and rows that start on 16 bytes, for which the descriptors hold
  if (a.w != nullptr || reinterpret_cast<uintptr_t>(a.in) % 16 != 0 ||
      a.in_stride * (dtype == DD_U8_I32 ? 1 : 4) % 16 != 0)
    return cudaErrorInvalidConfiguration;
#define X(T_, ...) \
  if (GS_IS(__VA_ARGS__)) return launch_t<T_, __VA_ARGS__>(cfg, a, s);
  if (dtype == DD_F32_F32) {
    DD_GSUM_F32(X)
  } else {
    DD_GSUM_U8(X)
  }
#undef X
  return cudaErrorInvalidConfiguration;
}

std::vector<TileConfig> gsum_menu(dd_dtype dtype) {
  std::vector<TileConfig> v;
#define X(T_, NC_, NS_, NP_, DPW_, SPL_, SS_, RB_, MB_)                                                            \
  v.push_back({Kind::GSum, NC_ * DPW_, 32 * SPL_, RB_, SS_, 32 * (NC_ + NS_ * NP_ + 1), SPL_, 0, NC_, \
               "gsum8_w" #NC_ "p" #NS_ "x" #NP_ "_d" #DPW_ "_s" #SPL_ "_r" #SS_ #RB_});
  if (dtype == DD_F32_F32) {
    DD_GSUM_F32(X)
  } else {
    DD_GSUM_U8(X)
  }
#undef X
  return v;
}

int gsum_smem_for(dd_dtype dtype, const TileConfig& cfg) {
  const int es = dtype == DD_U8_I32 ? 1 : 4, er = dtype == DD_U8_I32 ? 2 : 4;
  const int64_t n = kHeadBytes + (int64_t)cfg.cc * cfg.bd * 4 +
                    cfg.stages * (cfg.gs.desc_max + (int64_t)kGsGroup * (cfg.bt + cfg.gs.padp) * es) +
                    (int64_t)cfg.cc * cfg.gs.cap * er + (dtype == DD_U8_I32 ? (int64_t)cfg.pitch * cfg.bt * 4 : 0);
  return n > kMaxSmemPerBlock ? -1 : (int)n;
}

}  // namespace dd
