// Plans: the delay table of Eq. 1 on the host, its device copies, and the
// per-plan tile configuration menu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>

#include "dd_errors.h"
#include "dd_internal.h"

namespace dd {

std::vector<TileConfig> staged_menu(dd_dtype dtype);
std::vector<TileConfig> u8pk_menu(dd_dtype dtype);
std::vector<TileConfig> tmw6_menu(dd_dtype dtype);
std::vector<TileConfig> tmw9_menu(dd_dtype dtype);
std::vector<TileConfig> gsum_menu(dd_dtype dtype);
int u8pk_smem_for(const TileConfig& cfg, int pitch);
int staged_smem_for(dd_dtype dtype, int stages, int cc, int bd, int pitch);

// Eq. 1 (Section 2): delay in seconds of channel frequency f relative to the
// top of the band f_h is 4150 * DM * (1/f^2 - 1/f_h^2) (MHz); divided by the
// sampling time and rounded half up to a whole number of samples.  Evaluated
// in IEEE double, never in float: float flips entries that lie within 1e-6
// samples of a rounding boundary.
static dd_status compute_delay_table(dd_plan_s& p) {
  const double f_h = p.f_low + (double)(p.C - 1) * p.chan_bw;
  const double inv_fh2 = 1.0 / (f_h * f_h);
  p.delays.assign((size_t)p.n_dm * p.C, 0);
  for (int32_t i = 0; i < p.n_dm; ++i) {
    const double kdm = 4150.0 * (p.dm_first + (double)(p.dm_index0 + i) * p.dm_step);
    for (int32_t c = 0; c < p.C; ++c) {
      const double f = p.f_low + (double)c * p.chan_bw;
      const double samples = kdm * (1.0 / (f * f) - inv_fh2) / p.t_samp;
      const double r = std::floor(samples + 0.5);
      if (!(r >= 0.0) || r > 2147483647.0)
        return set_error(DD_ERR_ARG, "delay of channel %d at DM trial %d does not fit int32 (%.3g samples)", c,
                         i, samples);
      p.delays[(size_t)i * p.C + c] = (int32_t)r;
    }
  }
  return DD_OK;
}

// Largest (delay(c, i + bd - 1) - delay(c, i)) over channels and block starts i
// that are multiples of bd: the widest extra span a block of bd DM trials
// needs beyond its bt samples.  Trials past n_dm repeat the last one.
static int32_t block_spread(const dd_plan_s& p, int bd) {
  int32_t best = 0;
  for (int32_t i0 = 0; i0 < p.n_dm; i0 += bd) {
    const int32_t il = std::min(i0 + bd - 1, p.n_dm - 1);
    for (int32_t c = 0; c < p.C; ++c) {
      const int32_t s = p.delays[(size_t)il * p.C + c] - p.delays[(size_t)i0 * p.C + c];
      best = std::max(best, s);
    }
  }
  return best;
}

// Descriptor of (channel c, group of 6 trials starting at 6g), stored
// group-major ([g][c]: a block reads consecutive entries), for windows
// aligned down to 4 floats: x = delay of the group's first trial; y, z = the
// column of each trial's first sample in the window, (x & 3) + offset, one
// byte each (trials 0..3 in y, 4..5 in z); w = window width in floats,
// (x & 3) + 32 + the largest offset.  Returns the largest offset seen.
static int32_t build_hex_desc(const dd_plan_s& p, std::vector<int4>& desc) {
  const int32_t n_g = (p.n_dm + 5) / 6;
  desc.assign((size_t)p.C * n_g, int4{0, 0, 0, 0});
  int32_t worst = 0;
  for (int32_t c = 0; c < p.C; ++c) {
    for (int32_t g = 0; g < n_g; ++g) {
      const int32_t base = p.delays[(size_t)(6 * g) * p.C + c];
      const int32_t sh = base & 3;
      uint32_t packed[2] = {0, 0};
      int32_t mx = 0;
      for (int j = 0; j < 6; ++j) {
        const int32_t i = std::min(6 * g + j, p.n_dm - 1);
        const int32_t o = p.delays[(size_t)i * p.C + c] - base;
        mx = std::max(mx, o);
        packed[j / 4] |= (uint32_t)std::min(sh + o, 255) << (8 * (j % 4));
      }
      worst = std::max(worst, mx);
      desc[(size_t)g * p.C + c] = int4{base, (int)packed[0], (int)packed[1], sh + 32 + mx};
    }
  }
  return worst;
}

// Descriptor of (channel c, group of 9 trials starting at 9g), group-major
// ([g][c]), for windows that start at the 4-float boundary at or below the
// group's first sample: x = delay of the group's first trial; bytes 0..2 of
// y, z, w = the column of the first sample of trials 0..2, 3..5, 6..8 in the
// window, (x & 3) + offset (the warp reading trials 3p..3p+2 takes word p);
// byte 3 of y = the window's 4-float chunks, ceil(((x & 3) + 32 + largest
// offset) / 4).  Returns the largest offset seen.
static int32_t build_nine_desc(const dd_plan_s& p, std::vector<int4>& desc) {
  const int32_t n_g = (p.n_dm + 8) / 9;
  desc.assign((size_t)p.C * n_g, int4{0, 0, 0, 0});
  int32_t worst = 0;
  for (int32_t c = 0; c < p.C; ++c) {
    for (int32_t g = 0; g < n_g; ++g) {
      const int32_t base = p.delays[(size_t)(9 * g) * p.C + c];
      const int32_t sh = base & 3;
      uint32_t word[3] = {0, 0, 0};
      int32_t mx = 0;
      for (int j = 0; j < 9; ++j) {
        const int32_t i = std::min(9 * g + j, p.n_dm - 1);
        const int32_t o = p.delays[(size_t)i * p.C + c] - base;
        mx = std::max(mx, o);
        word[j / 3] |= (uint32_t)std::min(sh + o, 255) << (8 * (j % 3));
      }
      worst = std::max(worst, mx);
      const uint32_t nch = (uint32_t)std::min((sh + 32 + mx + 3) / 4, 255);
      desc[(size_t)g * p.C + c] = int4{base, (int)(word[0] | nch << 24), (int)word[1], (int)word[2]};
    }
  }
  return worst;
}

int32_t block_spread_of(const dd_plan_s& p, int bd) { return block_spread(p, bd); }

// Device memory of a plan's tables, from its host delay table alone: the
// table [n_dm][C], its transposed padded copy [C][n_dm_pad], the status word,
// and the 6- and 9-trial window descriptors where a group's offsets fit the
// Tensor-Memory windows (float plans).  finish_plan allocates exactly these;
// the footprint queries report the same numbers without allocating.
struct TableSizes {
  size_t delays = 0, delays_t = 0, status = sizeof(int), hex = 0, nine = 0, gsum = 0;
  int64_t total() const { return (int64_t)(delays + delays_t + status + hex + nine + gsum); }
};
using GsumTables = std::vector<std::pair<TileConfig, GsTable>>;

static double estimate_us(const dd_plan_s& p, const TileConfig& c);
static int best_config(const dd_plan_s& p, bool any_rows);

// The most patterns, by trials a block, with which sharing sums pays against the
// other kernels of the type (Apertif grid, uint8: 13.7 of 64 trials at 1024
// channels 1.39 ms against 2.09; about 20 at 512 the same as u8pk; float, whose
// other kernel on a transposed plan reads shared memory once an add, further).
// Below 192 channels nothing was gained at any size.
static double gs_max_patterns(const dd_plan_s& p, const TileConfig& c) {
  if (p.dtype == DD_F32_F32) return 32.0;
  if (p.C < 192) return 0.0;
  if (p.n_dm >= 512 && (c.bd != 64 || c.bt != 576)) return 0.0;  // the other shapes are for small launches
  return c.bd == 64 ? 18.0 : c.bd == 32 ? 14.0 : 8.0;
}

// The GSUM configurations a plan gets, with their descriptors.  Float forward
// plans get none: their kernels all add channel by channel, bit for bit the
// same, and GSUM adds eight channels first.
static GsumTables gsum_tables(const dd_plan_s& p) {
  GsumTables v;
  if (p.dtype == DD_F32_F32 && !p.grouped) return v;
  try {
    std::vector<TileConfig> cfgs;
    std::vector<GsTable> tables;
    for (TileConfig cfg : gsum_menu(p.dtype)) {
      const double most = gs_max_patterns(p, cfg);
      if (most <= 0.0) continue;
      const GsSample s = gsum_sample(p, cfg.bd, cfg.bt, most);
      if (s.patterns < 0.0 || s.patterns > most) continue;
      cfg.gs.patterns = (float)s.patterns;
      cfg.gs.samples = (float)s.samples;
      // the adjoint's plan is made by the first call that needs it: only a table it will use
      if (p.grouped && estimate_us(p, cfg) >= estimate_us(p, p.configs[best_config(p, false)])) continue;
      cfgs.push_back(cfg);
      tables.emplace_back();
      tables.back().bd = cfg.bd;
      tables.back().T = cfg.bt;
    }
    if (!tables.empty()) gsum_build(p, tables);
    for (size_t k = 0; k < tables.size(); ++k) {
      TileConfig& cfg = cfgs[k];
      GsTable& t = tables[k];
      if (!t.fits) continue;
      const int es = p.dtype == DD_U8_I32 ? 1 : 4, er = p.dtype == DD_U8_I32 ? 2 : 4;
      cfg.gs.padp = t.padp;
      cfg.gs.desc_max = t.desc_max;
      cfg.gs.cap = (int)t.cap;
      cfg.gs.reach = kGsGroup * (cfg.bt + t.padp) + cfg.cc * cfg.gs.cap * er / es;
      cfg.smem = gsum_smem_for(p.dtype, cfg);
      if (cfg.smem > 0) v.emplace_back(cfg, std::move(t));
    }
  } catch (const std::bad_alloc&) {  // the plan works without
    v.clear();
  }
  return v;
}

static TableSizes table_sizes(const dd_plan_s& p, const GsumTables& gsum) {
  TableSizes t;
  for (const auto& g : gsum) t.gsum += g.second.idx_bytes() + g.second.desc_bytes();
  const int64_t n_dm_pad = (p.n_dm + kDmPad - 1) / kDmPad * kDmPad;
  t.delays = (size_t)p.n_dm * p.C * 4;
  t.delays_t = (size_t)p.C * n_dm_pad * 4;
  if (p.dtype == DD_F32_F32) {
    // a group's largest offset is its last trial's delay less its first's
    if (block_spread(p, 6) <= kW6MaxOff) t.hex = (size_t)p.C * ((p.n_dm + 5) / 6) * sizeof(int4);
    if (block_spread(p, 9) <= kW9MaxOff) t.nine = (size_t)p.C * ((p.n_dm + 8) / 9) * sizeof(int4);
  }
  return t;
}

int64_t plan_in_stride(const dd_plan_s& p) {
  if (p.dtype == DD_U8_I32) return (p.n_in + 127) / 128 * 128;
  return tmw9_min_in_stride(p.n_in);
}

int64_t stream_buffer_bytes(const dd_plan_s& chunk_plan) {
  const int64_t elem = chunk_plan.dtype == DD_U8_I32 ? 1 : 4;
  return 2 * (int64_t)chunk_plan.C * plan_in_stride(chunk_plan) * elem;
}

void free_plan_device(dd_plan_s* p) {
  cudaFree(p->d_delays);
  cudaFree(p->d_delaysT);
  cudaFree(p->d_hex_desc);
  cudaFree(p->d_nine_desc);
  for (void* d : p->d_gs) cudaFree(d);
  p->d_gs.clear();
  cudaFree(p->d_status);
  cudaFree(p->h_dev_in);
  cudaFree(p->h_dev_out);
  cudaFree(p->h_dev_w);
  for (int k = 0; k < 5; ++k)
    if (p->h_streams[k]) cudaStreamDestroy(p->h_streams[k]);
  for (cudaEvent_t ev : p->h_events) cudaEventDestroy(ev);
  p->h_events.clear();
  cudaFree(p->adj_pad);
  cudaFree(p->adj_g);
  cudaFree(p->adj_wpart);
  if (p->adj) {
    free_plan_device(p->adj);
    delete p->adj;
    p->adj = nullptr;
  }
  p->d_delays = p->d_delaysT = nullptr;
  p->d_hex_desc = nullptr;
  p->d_nine_desc = nullptr;
  p->d_status = nullptr;
  p->h_dev_in = p->h_dev_out = nullptr;
  p->h_dev_w = nullptr;
  for (int k = 0; k < 5; ++k) p->h_streams[k] = nullptr;
  p->adj_pad = p->adj_g = nullptr;
  p->adj_wpart = nullptr;
  p->adj_wpart_floats = 0;
}

// Default configuration: the one whose time estimate is least.  The launch sizes
// decide between the kernels (40 tiles of TMW9 leave most SMs idle, and short
// chains of plain loads beat them), so the estimate is what was measured of
// each on this GPU (hence its 152 SMs, wherever the estimate is made), in
// microseconds per channel:
//   waves x (time of a block that shares its SM with as many as fill it), but no
//   less than the time of a block alone, plus what a launch costs.
//                      wave   alone   measured on (channels x trials x samples)
//   tmw9               0.303  0.303   1024 x 2048 x 20,000: 2.49 ms; x 64: 316 us
//   tmw6               0.331  0.331   1024 x 2048 x 20,000: 4.07 ms
//   staged d32 t512 c8 0.285  0.385   LOFAR beam 3.07 ms (d8 t1024 3.15); 107 x 2947 x 6576: 253 us
//   staged d16 t512    0.156  0.27    403 x 89 x 21,373: 140 us
//   staged d8 t1024    0.149  0.31    171 x 449 x 47,040: 478 us (d32 513)
//   staged d8 t512     0.078  0.187   126 x 21 x 77,585: 41 us (tmw9 48)
//   staged d8 t256     0.046  0.155   768 x 251 x 2414: 142 us (tmw9 239)
//   u8pk 32 trials     0.165  0.257   and 3.8 us per million outputs and 256 channels (its sums leave by
//                                     reading the output back): LOFAR 256 x 1024 x 50,000 650 us (16 trials 873)
//   u8pk 16 trials     0.108  0.142   167 x 1618 x 27,087: 414 us (32 trials 487); 16-channel chunks 0.112, 0.150
//   u8pk 1792 samples  0.11   0.149
//   u8pk 8 trials      0.075  0.104   182 x 92 x 5295: 23 us (16 trials 31)
// A staged wave costs the more the fewer there are (the ends of blocks overlap
// less), u8pk 32 trials 1.25 times as much where long spans leave one block an SM, and
// only pay from eight waves on (281 x 212 x 36,563: 254 us, 16 trials 165).
// Steep grids have spans much longer than their tiles.  What they cost is not the
// longer copies but the blocks that no longer fit an SM together: with one, each
// takes its own time (staged d8 t1024 0.30 a wave at any span from 9 to 17 KB,
// uint8 and float), with a few a little more than their share of it.  Timed on
// 1,020 random beams at 0 to 256 times the surveys' DM steps, the choice is
// within 2 % of the best of the menu on average and within 5 % of the fixed
// preference list it replaced on every one (LOFAR 30 x 477 x 66,978 at 0.32, uint8:
// staged d8 t1024 161 us, plain 445; Apertif 447 x 223 x 17,992 at 8, float:
// 325 us, d8 t512 553).
// The plain kernel needs 0.030 a channel (uint8; float less), or 2.4 T adds/s where
// that is more, with eight channels' worth of time for each output (float LOFAR
// 319 x 750 x 6048 at 0.64: 530 us in blocks of 256, 666 in blocks of 128; 1024 x 2 x
// 20,000: 49 and 26).
// GSUM's times grow with the samples of the rows its blocks make (a block's
// patterns times the row's length; 11,000 a group on the Apertif beam), which the
// row makers may need longer for than the adding: 64 trials 1.39 ms there (u8pk 2.09),
// 32 trials 98 us on 1024 x 64 x 20,000 (u8pk 145), 16 trials 75 us on
// 768 x 251 x 2414 (u8pk 85); float, on the Apertif beam's adjoint: 3.4 ms (staged 7.1).
static double estimate_us(const dd_plan_s& p, const TileConfig& c) {
  constexpr double kNever = 1e30;
  const double C = p.C, outputs = p.n_dm * (double)p.n_out;
  const double tiles = std::ceil((double)p.n_dm / c.bd) * std::ceil((double)p.n_out / c.bt);
  const double waves = std::ceil(tiles / 152.0);
  auto time = [&](double wave, double alone) { return 6.0 + C * std::max(alone, waves * wave); };
  // blocks whose spans fit an SM together: fewer than it takes to fill its time
  // cost a block's own time each
  const double fit = std::max(1.0, std::floor(228.0 * 1024 / (c.smem + 1024)));
  auto spans = [&](double wave, double alone) {
    return time(std::max(wave, fit > 1.0 ? 1.15 * alone / fit : alone), alone);
  };
  const bool u8 = p.dtype == DD_U8_I32;
  switch (c.kind) {
    case Kind::Naive:
      // (launches of more threads than fit the SMs at once: blocks of 256, the same
      // on 200 random ones on average, 5 to 20 % less on steep float ones of many
      // channels; small ones up to 1.9 times as much)
      if (c.threads != (outputs > 152.0 * 2048 ? 256 : 128)) return kNever;
      return 5.0 + std::max(0.030 * C, (C + 8.0) * outputs / 2.4e6);
    case Kind::TmW9:
      return 1.0 + time(0.303, 0.303);
    case Kind::TmW6:
      return 1.0 + time(0.331, 0.331);
    case Kind::Staged:
      if (c.bd == 32 && c.bt == 512 && c.cc == 8 && !u8) return spans(0.285 + 0.086 / waves, 0.385);
      if (c.bd == 16 && c.bt == 512) return spans(0.156 + 0.078 / waves, 0.27);
      if (c.bd == 8 && c.bt == 1024) return spans(0.149 + 0.042 / waves, 0.31);
      if (c.bd == 8 && c.bt == 512) return spans(0.078 + 0.057 / waves, 0.187);
      if (c.bd == 8 && c.bt == 256)  // long spans cost its short tiles most (293 x 1081 x 1064, LOFAR: 0.067)
        return spans((0.046 + 0.045 / waves) * (1.0 + 0.22 * (c.pitch - c.bt) / c.bt), 0.155);
      return kNever;
    case Kind::U8Pk: {
      const double one = 2 * (c.smem + 1024) > 228 * 1024 ? 1.25 : 1.0;  // one block an SM
      if (c.bd == 32 && c.stages == 3)
        return waves < 8.0 ? kNever
                           : time(0.165 * one * (c.cc == 16 ? 1.03 : 1.0), 0.257) +
                                 3.8e-6 * outputs * std::ceil(C / 256.0);
      if (c.bd == 16 && c.bt == 896) return spans(c.cc == 32 ? 0.108 : 0.112, c.cc == 32 ? 0.142 : 0.150) + 0.6e-6 * outputs;
      if (c.bt == 1792) return spans(c.bd == 8 && c.threads == 512 ? 0.115 : 0.11, 0.149) + 0.85e-6 * outputs;
      if (c.bd == 8 && c.threads == 128)  // two blocks an SM
        return spans(0.15 * std::ceil(waves / 2.0) / waves, 0.104) + 0.5e-6 * outputs;
      return kNever;
    }
    case Kind::GSum: {
      if (c.gs.patterns > 0.9 * std::min(c.bd, p.n_dm)) return kNever;  // hardly two trials share one
      if (!u8) return time(0.12 + 0.0065 * c.gs.patterns, 0.20);
      const double rows = 1e-3 * c.gs.samples;  // thousands of row samples a group
      // adding the rows up; making them, if that takes longer; a block alone
      auto gsum = [&](double add, double make, double alone) {
        return 6.0 + C * std::max({waves * add, std::ceil(waves / (c.bd == 16 ? 2.0 : 1.0)) * make * rows, alone});
      };
      if (c.bd == 64 && c.bt == 576) return gsum(0.085 + 0.0090 * rows, 0.0163, 0.103);
      if (c.bd == 64) return gsum(0.088 + 0.0059 * rows, 0.0149, 0.098);
      if (c.bd == 32) return gsum(0.079 + 0.0029 * rows, 0.0152, 0.083);
      return gsum(0.044 + 0.0065 * rows, 0.0293, 0.080);
    }
    default:
      return kNever;
  }
}

// Configurations by their estimate, then the rest of the menu in its order.
std::vector<int> config_preference_order(const dd_plan_s& p) {
  std::vector<int> order(p.configs.size());
  std::vector<double> est(p.configs.size());
  for (size_t j = 0; j < order.size(); ++j) {
    order[j] = (int)j;
    est[j] = estimate_us(p, p.configs[j]);
    // the plain kernel's other block sizes last
    if (p.configs[j].kind == Kind::Naive && est[j] >= 1e30) est[j] *= 2.0;
  }
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return est[x] < est[y]; });
  return order;
}

static int best_config(const dd_plan_s& p, bool any_rows) {
  for (int j : config_preference_order(p))
    if (!any_rows || takes_any_rows(p.configs[j])) return j;
  return 0;
}

// Everything a plan derives from its delay table (p->delays [n_dm][C], rows
// non-decreasing along the trial index for every channel): sizes, device
// copies of the table and descriptors, and the configuration menu.
dd_status finish_plan(dd_plan_s* p) {
  p->max_delay = *std::max_element(p->delays.begin(), p->delays.end());
  p->n_in = p->n_out + p->max_delay;
  p->n_dm_pad = (p->n_dm + kDmPad - 1) / kDmPad * kDmPad;

  if (cudaGetDevice(&p->device) != cudaSuccess) return set_cuda_error("dd_plan: cudaGetDevice");
  // transposed, padded copy: [C][n_dm_pad], trials past n_dm repeat the last
  std::vector<int32_t> dT((size_t)p->C * p->n_dm_pad);
  for (int32_t c = 0; c < p->C; ++c)
    for (int32_t i = 0; i < p->n_dm_pad; ++i)
      dT[(size_t)c * p->n_dm_pad + i] = p->delays[(size_t)std::min(i, p->n_dm - 1) * p->C + c];
  const TableSizes sizes = table_sizes(*p, {});
  const size_t bytes_d = sizes.delays, bytes_dT = sizes.delays_t;
  cudaError_t e = cudaMalloc(&p->d_delays, bytes_d);
  if (e == cudaSuccess) e = cudaMalloc(&p->d_delaysT, bytes_dT);
  if (e == cudaSuccess) e = cudaMalloc(&p->d_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpy(p->d_delays, p->delays.data(), bytes_d, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(p->d_delaysT, dT.data(), bytes_dT, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(p->d_status, 0, sizeof(int));
  if (e != cudaSuccess) {
    free_plan_device(p);
    return e == cudaErrorMemoryAllocation ? set_error(DD_ERR_NOMEM, "dd_plan: device allocation failed")
                                          : set_cuda_error("dd_plan: upload", e);
  }
  p->device_bytes = (int64_t)(bytes_d + bytes_dT + sizeof(int));
  // 6-trial descriptors, only where the windows fit (float plans, offsets <= 31)
  bool hex_ok = false;
  if (sizes.hex > 0) {
    std::vector<int4> desc6;
    if (build_hex_desc(*p, desc6) <= kW6MaxOff) {
      const size_t bytes6 = desc6.size() * sizeof(int4);
      e = cudaMalloc(&p->d_hex_desc, bytes6);
      if (e == cudaSuccess) e = cudaMemcpy(p->d_hex_desc, desc6.data(), bytes6, cudaMemcpyHostToDevice);
      if (e != cudaSuccess) {
        free_plan_device(p);
        return e == cudaErrorMemoryAllocation ? set_error(DD_ERR_NOMEM, "dd_plan: device allocation failed")
                                              : set_cuda_error("dd_plan: upload", e);
      }
      p->device_bytes += (int64_t)bytes6;
      hex_ok = true;
    }
  }
  bool nine_ok = false;
  if (sizes.nine > 0) {
    std::vector<int4> desc9;
    if (build_nine_desc(*p, desc9) <= kW9MaxOff) {
      const size_t bytes9 = desc9.size() * sizeof(int4);
      e = cudaMalloc(&p->d_nine_desc, bytes9);
      if (e == cudaSuccess) e = cudaMemcpy(p->d_nine_desc, desc9.data(), bytes9, cudaMemcpyHostToDevice);
      if (e != cudaSuccess) {
        free_plan_device(p);
        return e == cudaErrorMemoryAllocation ? set_error(DD_ERR_NOMEM, "dd_plan: device allocation failed")
                                              : set_cuda_error("dd_plan: upload", e);
      }
      p->device_bytes += (int64_t)bytes9;
      nine_ok = true;
    }
  }
  // configuration menu, filtered by what this geometry allows
  const int V = p->dtype == DD_U8_I32 ? 16 : 4;
  for (TileConfig cfg : staged_menu(p->dtype)) {
    if (cfg.kind == Kind::Staged) {
      const int64_t spread = block_spread(*p, cfg.bd);
      const int64_t pitch = (cfg.bt + spread + 2 * V + V - 1) / V * V;
      if (pitch > (int64_t)1 << 20) continue;
      cfg.pitch = (int)pitch;
      cfg.smem = staged_smem_for(p->dtype, cfg.stages, cfg.cc, cfg.bd, cfg.pitch);
      if (cfg.smem > kMaxSmemPerBlock) continue;
      if ((p->n_dm + cfg.bd - 1) / cfg.bd > 65535) continue;
    }
    p->configs.push_back(cfg);
  }
  for (TileConfig cfg : u8pk_menu(p->dtype)) {
    const int64_t spread = block_spread(*p, cfg.bd);
    // + 32: a lane reads 32 bytes from a word-aligned start at or before its first sample
    const int64_t pitch = (cfg.bt + spread + 2 * V + 32 + V - 1) / V * V;
    if (pitch > (int64_t)1 << 20) continue;
    cfg.pitch = (int)pitch;
    cfg.smem = u8pk_smem_for(cfg, cfg.pitch);
    if (cfg.smem > kMaxSmemPerBlock) continue;
    if ((p->n_dm + cfg.bd - 1) / cfg.bd > 65535) continue;
    p->configs.push_back(cfg);
  }
  if (hex_ok) {
    for (TileConfig cfg : tmw6_menu(p->dtype)) {
      if ((p->n_out + cfg.bt - 1) / cfg.bt > 65535) continue;  // time tiles are the grid's y
      p->configs.push_back(cfg);
    }
  }
  if (nine_ok) {
    for (TileConfig cfg : tmw9_menu(p->dtype)) {
      if ((p->n_out + cfg.bt - 1) / cfg.bt > 65535) continue;
      p->configs.push_back(cfg);
    }
  }
  for (auto& [cfg, t] : gsum_tables(*p)) {
    void* d[2] = {nullptr, nullptr};
    const void* h[2] = {t.idx.data(), t.desc.data()};
    const size_t n[2] = {t.idx_bytes(), t.desc_bytes()};
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaMalloc(&d[k], n[k]);
    if (e == cudaErrorMemoryAllocation) {  // the plan works without
      cudaGetLastError();
      cudaFree(d[0]);
      e = cudaSuccess;
      continue;
    }
    p->d_gs.insert(p->d_gs.end(), d, d + 2);
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaMemcpy(d[k], h[k], n[k], cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      free_plan_device(p);
      return set_cuda_error("dd_plan: upload", e);
    }
    p->device_bytes += (int64_t)(n[0] + n[1]);
    cfg.gs.idx = static_cast<const uint2*>(d[0]);
    cfg.gs.desc = static_cast<const uint4*>(d[1]);
    if ((p->n_out + cfg.bt - 1) / cfg.bt <= 65535) p->configs.push_back(cfg);
  }
  p->selected = best_config(*p, false);
  // for inputs whose layout the selected one cannot take (TMW9 and TMW6 need
  // spare samples or 128-byte rows, most others rows that start on 16 bytes)
  p->fallback = best_config(*p, true);
  return DD_OK;
}

}  // namespace dd

using namespace dd;

static dd_status check_plan_args(int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                                 double dm_first, double dm_step, int32_t n_dm) {
  if (channels <= 0) return set_error(DD_ERR_ARG, "channels must be > 0 (got %d)", channels);
  if (!(f_low_mhz > 0.0) || !std::isfinite(f_low_mhz)) return set_error(DD_ERR_ARG, "f_low must be > 0 MHz");
  if (!(chan_bw_mhz > 0.0) || !std::isfinite(chan_bw_mhz)) return set_error(DD_ERR_ARG, "chan_bw must be > 0 MHz");
  if (!(t_samp_s > 0.0) || !std::isfinite(t_samp_s)) return set_error(DD_ERR_ARG, "t_samp must be > 0 s");
  if (!(dm_first >= 0.0) || !std::isfinite(dm_first)) return set_error(DD_ERR_ARG, "dm_first must be >= 0");
  if (!(dm_step >= 0.0) || !std::isfinite(dm_step)) return set_error(DD_ERR_ARG, "dm_step must be >= 0");
  if (n_dm <= 0) return set_error(DD_ERR_ARG, "n_dm must be > 0 (got %d)", n_dm);
  if ((int64_t)channels * n_dm > (int64_t)1 << 31)
    return set_error(DD_ERR_ARG, "delay table of %lld entries is too large", (long long)channels * n_dm);
  return DD_OK;
}

extern "C" dd_status dd_delay_table(int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                                    double dm_first, double dm_step, int32_t n_dm, int32_t* host_out) {
  return dd_delay_table_dm_range(channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, 0, n_dm, host_out);
}

extern "C" dd_status dd_delay_table_dm_range(int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                                             double dm_first, double dm_step, int32_t dm_index0, int32_t n_dm,
                                             int32_t* host_out) {
  clear_error();
  if (!host_out) return set_error(DD_ERR_ARG, "dd_delay_table: host_out is NULL");
  dd_status st = check_plan_args(channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, n_dm);
  if (st != DD_OK) return st;
  if (dm_index0 < 0 || (int64_t)dm_index0 + n_dm > 2147483647LL)
    return set_error(DD_ERR_ARG, "dd_delay_table: first trial index %d out of range", dm_index0);
  dd_plan_s p;
  p.C = channels;
  p.n_dm = n_dm;
  p.f_low = f_low_mhz;
  p.chan_bw = chan_bw_mhz;
  p.t_samp = t_samp_s;
  p.dm_first = dm_first;
  p.dm_step = dm_step;
  p.dm_index0 = dm_index0;
  st = compute_delay_table(p);
  if (st != DD_OK) return st;
  std::memcpy(host_out, p.delays.data(), p.delays.size() * sizeof(int32_t));
  return DD_OK;
}

extern "C" dd_status dd_plan(dd_plan_t* out, int32_t channels, double f_low_mhz, double chan_bw_mhz,
                             double t_samp_s, double dm_first, double dm_step, int32_t n_dm, int64_t n_out,
                             dd_dtype dtype) {
  return dd_plan_dm_range(out, channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, 0, n_dm, n_out, dtype);
}

extern "C" dd_status dd_plan_dm_range(dd_plan_t* out, int32_t channels, double f_low_mhz, double chan_bw_mhz,
                                      double t_samp_s, double dm_first, double dm_step, int32_t dm_index0,
                                      int32_t n_dm, int64_t n_out, dd_dtype dtype) {
  clear_error();
  if (!out) return set_error(DD_ERR_ARG, "dd_plan: out is NULL");
  dd_status chk = check_plan_args(channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, n_dm);
  if (chk != DD_OK) return chk;
  if (dm_index0 < 0 || (int64_t)dm_index0 + n_dm > 2147483647LL)
    return set_error(DD_ERR_ARG, "dd_plan_dm_range: first trial index %d out of range", dm_index0);
  if (n_out <= 0) return set_error(DD_ERR_ARG, "dd_plan: n_out must be > 0");
  if (dtype != DD_U8_I32 && dtype != DD_F32_F32) return set_error(DD_ERR_ARG, "dd_plan: unknown dtype %d", (int)dtype);
  if (dtype == DD_U8_I32 && (int64_t)channels * 255 > 2147483647LL)
    return set_error(DD_ERR_ARG, "dd_plan: %d channels of uint8 overflow int32 sums", channels);

  dd_plan_s* p = new (std::nothrow) dd_plan_s();
  if (!p) return set_error(DD_ERR_NOMEM, "dd_plan: host allocation failed");
  p->C = channels;
  p->n_dm = n_dm;
  p->n_out = n_out;
  p->f_low = f_low_mhz;
  p->chan_bw = chan_bw_mhz;
  p->t_samp = t_samp_s;
  p->dm_first = dm_first;
  p->dm_step = dm_step;
  p->dm_index0 = dm_index0;
  p->dtype = dtype;
  dd_status st = compute_delay_table(*p);
  if (st != DD_OK) {
    delete p;
    return st;
  }
  st = finish_plan(p);
  if (st != DD_OK) {
    delete p;
    return st;
  }
  apply_tune_db(p);
  *out = p;
  return DD_OK;
}

// A host-only plan of the given geometry with its delay table (no device
// memory), for the footprint queries.
static dd_status host_plan(dd_plan_s& p, int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                           double dm_first, double dm_step, int32_t n_dm, int64_t n_out, dd_dtype dtype) {
  dd_status st = check_plan_args(channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, n_dm);
  if (st != DD_OK) return st;
  if (dtype != DD_U8_I32 && dtype != DD_F32_F32) return set_error(DD_ERR_ARG, "unknown dtype %d", (int)dtype);
  p.C = channels;
  p.n_dm = n_dm;
  p.n_out = n_out;
  p.f_low = f_low_mhz;
  p.chan_bw = chan_bw_mhz;
  p.t_samp = t_samp_s;
  p.dm_first = dm_first;
  p.dm_step = dm_step;
  p.dtype = dtype;
  st = compute_delay_table(p);
  if (st != DD_OK) return st;
  p.max_delay = *std::max_element(p.delays.begin(), p.delays.end());
  p.n_in = p.n_out + p.max_delay;
  return DD_OK;
}

extern "C" dd_status dd_plan_footprint(int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                                       double dm_first, double dm_step, int32_t n_dm, dd_dtype dtype,
                                       int64_t* device_bytes) {
  clear_error();
  if (!device_bytes) return set_error(DD_ERR_ARG, "dd_plan_footprint: device_bytes is NULL");
  dd_plan_s p;
  dd_status st = host_plan(p, channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, n_dm, 1, dtype);
  if (st != DD_OK) return st;
  *device_bytes = table_sizes(p, gsum_tables(p)).total();
  return DD_OK;
}

extern "C" dd_status dd_stream_footprint(int32_t channels, double f_low_mhz, double chan_bw_mhz, double t_samp_s,
                                         double dm_first, double dm_step, int32_t n_dm, int64_t chunk_len,
                                         dd_dtype dtype, int64_t* device_bytes) {
  clear_error();
  if (!device_bytes) return set_error(DD_ERR_ARG, "dd_stream_footprint: device_bytes is NULL");
  if (chunk_len <= 0) return set_error(DD_ERR_ARG, "dd_stream_footprint: chunk_len must be > 0");
  dd_plan_s p;  // the stream's own plan: the same geometry, n_out = chunk_len
  dd_status st = host_plan(p, channels, f_low_mhz, chan_bw_mhz, t_samp_s, dm_first, dm_step, n_dm, chunk_len, dtype);
  if (st != DD_OK) return st;
  *device_bytes = table_sizes(p, gsum_tables(p)).total() + stream_buffer_bytes(p);
  return DD_OK;
}

extern "C" dd_status dd_plan_destroy(dd_plan_t plan) {
  clear_error();
  if (!plan) return DD_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != plan->device) cudaSetDevice(plan->device);
  free_plan_device(plan);
  if (prev >= 0 && prev != plan->device) cudaSetDevice(prev);
  delete plan;
  return DD_OK;
}

extern "C" dd_status dd_plan_info(dd_plan_t plan, int64_t* n_in, int32_t* max_delay, int64_t* device_bytes) {
  clear_error();
  if (!plan) return set_error(DD_ERR_ARG, "dd_plan_info: plan is NULL");
  if (n_in) *n_in = plan->n_in;
  if (max_delay) *max_delay = plan->max_delay;
  if (device_bytes) *device_bytes = plan->device_bytes;
  return DD_OK;
}

extern "C" dd_status dd_plan_in_stride(dd_plan_t plan, int64_t* in_row_stride) {
  clear_error();
  if (!plan || !in_row_stride) return set_error(DD_ERR_ARG, "dd_plan_in_stride: NULL argument");
  *in_row_stride = plan_in_stride(*plan);
  return DD_OK;
}

extern "C" dd_status dd_plan_delays(dd_plan_t plan, int32_t* host_out) {
  clear_error();
  if (!plan || !host_out) return set_error(DD_ERR_ARG, "dd_plan_delays: NULL argument");
  std::memcpy(host_out, plan->delays.data(), plan->delays.size() * sizeof(int32_t));
  return DD_OK;
}

extern "C" dd_status dd_plan_num_configs(dd_plan_t plan, int32_t* n) {
  clear_error();
  if (!plan || !n) return set_error(DD_ERR_ARG, "dd_plan_num_configs: NULL argument");
  *n = (int32_t)plan->configs.size();
  return DD_OK;
}

extern "C" const char* dd_plan_config_name(dd_plan_t plan, int32_t k) {
  if (!plan || k < 0 || k >= (int32_t)plan->configs.size()) return nullptr;
  return plan->configs[k].name.c_str();
}

extern "C" dd_status dd_plan_select_config(dd_plan_t plan, int32_t k) {
  clear_error();
  if (!plan) return set_error(DD_ERR_ARG, "dd_plan_select_config: plan is NULL");
  if (k < 0 || k >= (int32_t)plan->configs.size())
    return set_error(DD_ERR_ARG, "dd_plan_select_config: config %d out of range [0, %zu)", k, plan->configs.size());
  plan->selected = k;
  plan->chosen_by = ChosenBy::Caller;
  return DD_OK;
}

extern "C" dd_status dd_plan_selected_config(dd_plan_t plan, int32_t* k) {
  clear_error();
  if (!plan || !k) return set_error(DD_ERR_ARG, "dd_plan_selected_config: NULL argument");
  *k = plan->selected;
  return DD_OK;
}

extern "C" dd_status dd_plan_device_status(dd_plan_t plan, int32_t* code) {
  clear_error();
  if (!plan || !code) return set_error(DD_ERR_ARG, "dd_plan_device_status: NULL argument");
  int v = 0;
  cudaError_t e = cudaMemcpy(&v, plan->d_status, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return set_cuda_error("dd_plan_device_status", e);
  *code = v;
  if (v != 0) {
    cudaMemset(plan->d_status, 0, sizeof(int));
    return set_error(DD_ERR_STATE, "a kernel of this plan reported device error %d (1 = bounded wait expired)", v);
  }
  return DD_OK;
}
