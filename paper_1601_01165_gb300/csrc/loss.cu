// Boxcar-8 S/N detection loss over a dedispersed block, and its gradient.
//
// Not part of the paper: this is the loss of the differentiable
// configuration (dedisperse -> 8-sample boxcar -> maximum S/N).  Per row i:
// b[t] = sum_{k<8} x[i][t+k], mean m and population sd s of b over
// t < nb = n_cols - 7, z[t] = (b[t] - m) / s.  loss = -max_{i,t} z (first on
// ties).  For the best row i*, t*:
//   d z[t*] / d b[t] = ((t == t*) - 1/nb) / s - z[t*] z[t] / (nb s)
//   d loss / d x[i*][u] = -sum over t in [u-7, u] of d z[t*] / d b[t].
// Each thread sums in two-float arithmetic (about 48 bits), each block in
// double; each row is one block with a fixed reduction tree.
#include <cuda_runtime.h>

#include <cfloat>
#include <mutex>

#include "dd_errors.h"
#include "dd_internal.h"

namespace dd {

constexpr int kBox = 8;

struct __align__(16) RowStat {
  double z;      // best S/N in the row (-inf if the row is constant)
  double mean;
  double sd;
  int64_t t;     // boxcar start of the best S/N
};

// Row i's statistics are eight words at stats + i * stride: in a scratch array,
// or, when a gradient is asked for, in the first eight samples of its row
// (cleared again with the gradient's own row), which needs no allocation.
__device__ __forceinline__ void put_stat(float* at, const RowStat& r) {
  static_assert(sizeof(RowStat) == 8 * sizeof(float), "eight words, the shortest row");
  const int4* v = reinterpret_cast<const int4*>(&r);
  const int w[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
  for (int k = 0; k < 8; ++k) at[k] = __int_as_float(w[k]);
}
__device__ __forceinline__ RowStat get_stat(const float* at) {
  int w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) w[k] = __float_as_int(at[k]);
  RowStat r;
  r.z = __hiloint2double(w[1], w[0]);
  r.mean = __hiloint2double(w[3], w[2]);
  r.sd = __hiloint2double(w[5], w[4]);
  r.t = (int64_t)((uint64_t)(uint32_t)w[7] << 32 | (uint32_t)w[6]);
  return r;
}

__device__ __forceinline__ double boxcar(const float* row, int64_t t) {
  double b = 0.0;
#pragma unroll
  for (int k = 0; k < kBox; ++k) b += (double)__ldg(row + t + k);
  return b;
}

template <int NT>
__device__ double block_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = NT / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

// Two-float ("double-float") numbers: h + l with |l| <= ulp(h) / 2, about 48
// significant bits.  Double arithmetic is slow on this GPU's SMs; these
// sums use a few single-precision operations each (Knuth's two-sum, Dekker's
// fast two-sum and an FMA-based exact product), with explicit round-to-nearest
// intrinsics so that the compiler neither fuses nor reorders them.
struct DF {
  float h, l;
};

__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ DF fast_two_sum(float a, float b) {  // |a| >= |b| or a == 0
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ DF df_add_f(DF a, float b) {
  const DF s = two_sum(a.h, b);
  return fast_two_sum(s.h, __fadd_rn(s.l, a.l));
}

__device__ __forceinline__ DF df_add(DF a, DF b) {
  const DF s = two_sum(a.h, b.h);
  const DF t = two_sum(a.l, b.l);
  const DF u = fast_two_sum(s.h, __fadd_rn(s.l, t.h));
  return fast_two_sum(u.h, __fadd_rn(u.l, t.l));
}

// The same for the boxcars, where a.l + b.l needs no exact error: two
// operations instead of nine.  The result is within 2^-47 (|a| + |b|), and
// exact wherever |a.l + b.l| fits 24 bits of the operands' common unit.  (A
// boxcar takes two of these, where one sample added after another rounds the
// low parts six times.)
__device__ __forceinline__ DF df_add_fast(DF a, DF b) {
  const DF s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

// d * d for a two-float d, as a two-float (the low part's square is dropped)
__device__ __forceinline__ DF df_sqr(DF d) {
  const float p = __fmul_rn(d.h, d.h);
  const float e = __fmaf_rn(d.h, d.h, -p);
  return fast_two_sum(p, __fmaf_rn(__fmul_rn(2.0f, d.h), d.l, e));
}

__device__ __forceinline__ DF df_of(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ double df_value(DF a) { return (double)a.h + (double)a.l; }

// a > b for normalised two-floats
__device__ __forceinline__ bool df_gt(DF a, DF b) { return a.h > b.h || (a.h == b.h && a.l > b.l); }

// The boxcars of a thread's K consecutive starts, from x[0 .. K + 7): pairs,
// fours, eights, each shared by the boxcars that need it (one add of floats
// and two of two-floats per start, against eight adds for a boxcar summed by
// itself).  Exact while the values' nonzero magnitudes lie within a factor of
// about 2^21: 48 bits hold the sum of eight 24-bit significands spread that far.
// visit(k, boxcar) in order of k.
template <int K, typename F>
__device__ __forceinline__ void boxcars(const float* x, F visit) {
  DF p2[6];  // pairs starting at the last six samples, then fours likewise
  DF p4[4];
#pragma unroll
  for (int u = 0; u < K + 6; ++u) {
    const DF two = two_sum(x[u], x[u + 1]);
    if (u >= 2) {
      const DF four = df_add_fast(p2[(u - 2) % 6], two);  // starts at u - 2
      if (u >= 6) visit(u - 6, df_add_fast(p4[(u - 6) % 4], four));
      p4[(u - 2) % 4] = four;
    }
    p2[u % 6] = two;
  }
}

// One block per row: mean, sd, best S/N and where it is; with ZERO the block
// also clears the row of the gradient while it computes.
//
// Instruction issue bounds it (77 % of the slots; 144 instructions a sample, where
// reading and clearing a 2048 x 20,000 block of 164 MB take 24 us each), so a
// row is passed over twice with as little as each needs:
//  1. the sum of the samples, which gives the boxcars' (a sample counts in
//     eight of them, at the row's ends in fewer);
//  2. from tiles of the row in shared memory, each thread's K consecutive
//     boxcars: the squares about the mean and the largest boxcar (K odd: the
//     lanes' reads hit distinct banks).
// Threads sum in two-float arithmetic, the block in double.  S/N is monotonic
// in the boxcar, so the best S/N is (b_max - mean) / sd, and the first start
// with that S/N lies among those whose boxcar is within rounding of b_max:
// only a thread that has another boxcar that close goes over its starts again
// (a different start only when two sums round to one S/N).
// 2048 x 20,000 with the gradient: the whole call 226 us, nearly all of it this
// kernel (before: 493, every boxcar summed by itself in each of three passes,
// the clearing after them, and 0.1 ms for the one row of the gradient).
template <int NT, int K, bool ZERO>
__global__ void __launch_bounds__(NT) snr_rows_kernel(const float* __restrict__ x, int64_t stride, int64_t n_cols,
                                                      float* stats, int64_t stats_stride, float* grad,
                                                      int64_t grad_stride) {
  constexpr int TILE = NT * K;
  __shared__ float tile[TILE + kBox - 1];
  __shared__ double red[NT];
  __shared__ int64_t tbest[NT];
  const int i = blockIdx.x, tid = threadIdx.x;
  const float* row = x + (int64_t)i * stride;
  const int64_t nb = n_cols - kBox + 1;

  // pass 1: the sum of the boxcars (a sample u is in min(u + 1, 8, n_cols - u, nb) of them)
  double sum = 0.0;
  if (nb < kBox) {
    // Few starts share most of their samples, and may differ by less than the
    // boxcars' own rounding: their mean is that of the boxcars as pass 2 has
    // them (one start has no deviation, two have S/N 1).
    if (tid < nb) boxcars<1>(row + tid, [&](int, DF b) { sum = df_value(b); });
  } else {
    DF s4[4] = {};
    int64_t u = tid;
    for (; u + 3 * NT < n_cols; u += 4 * NT) {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = __ldg(row + u + k * NT);
#pragma unroll
      for (int k = 0; k < 4; ++k) s4[k] = df_add_f(s4[k], v[k]);
    }
    for (; u < n_cols; u += NT) s4[0] = df_add_f(s4[0], __ldg(row + u));
    sum = (double)kBox * df_value(df_add(df_add(s4[0], s4[1]), df_add(s4[2], s4[3])));
    for (int64_t e = tid; e < 2 * (kBox - 1); e += NT) {  // the ends: count the missing ones off
      const int64_t at = e < kBox - 1 ? e : n_cols - 1 - (e - (kBox - 1));
      sum -= (double)(kBox - min(min(at + 1, n_cols - at), (int64_t)kBox)) * (double)__ldg(row + at);
    }
  }
  const double mean = block_sum<NT>(sum, red) / (double)nb;

  // pass 2: squares about the mean, and the largest boxcar of each thread (its first)
  const DF neg_mean = df_of(-mean);
  DF v{0.0f, 0.0f}, bmax{-FLT_MAX, 0.0f}, before{-FLT_MAX, 0.0f};  // `before`: the largest at earlier starts
  int at = -1;     // its place among this thread's starts, tile by tile
  int first = 0;   // the tile's first place
  for (int64_t base = 0; base < nb; base += TILE, first += K) {
    const int64_t len = min((int64_t)(TILE + kBox - 1), n_cols - base);
    for (int64_t k = tid; k < len; k += NT) tile[k] = __ldg(row + base + k);
    if constexpr (ZERO) {
      // (the last tile also clears the samples past the last start)
      float* gr = grad + (int64_t)i * grad_stride + base;
      const int64_t glen = base + TILE < nb ? (int64_t)TILE : n_cols - base;
      for (int64_t k = tid; k < glen; k += NT) gr[k] = 0.0f;
    }
    __syncthreads();
    const int64_t t0 = base + (int64_t)tid * K;
    const int n = (int)max((int64_t)0, min((int64_t)K, nb - t0));
    auto visit = [&](int k, DF b) {
      if (k < n) {
        // (the whole sums: where b is close to a large mean, nothing but the
        // low parts' exact sum is left of the difference)
        v = df_add(v, df_sqr(df_add(b, neg_mean)));
        if (at < 0 || df_gt(b, bmax)) {  // t increases, so the first maximum is kept
          before = bmax;
          bmax = b;
          at = first + k;
        }
      }
    };
    if (n > 0) boxcars<K>(tile + tid * K, visit);
    __syncthreads();
  }
  const double sd = sqrt(block_sum<NT>(df_value(v), red) / (double)nb);

  // the row's largest boxcar, its first start
  const double mine = df_value(bmax);
  const int64_t tmax = at < 0 ? -1 : (int64_t)(at / K) * TILE + (int64_t)tid * K + at % K;
  red[tid] = mine;
  tbest[tid] = tmax;
  __syncthreads();
  for (int h = NT / 2; h > 0; h >>= 1) {
    if (tid < h) {
      const double bo = red[tid + h];
      const int64_t to = tbest[tid + h];
      if (to >= 0 && (tbest[tid] < 0 || bo > red[tid] || (bo == red[tid] && to < tbest[tid]))) {
        red[tid] = bo;
        tbest[tid] = to;
      }
    }
    __syncthreads();
  }
  const double b_top = red[0];
  const int64_t t_top = tbest[0];
  __syncthreads();
  if (!(sd > 0.0)) {
    if (tid == 0) put_stat(stats + i * stats_stride, RowStat{-DBL_MAX, mean, sd, -1});
    return;
  }
  const double z_top = (b_top - mean) / sd;

  // the first start with the same S/N, if it is before t_top
  const double b_cut = b_top - 1e-12 * (fabs(b_top - mean) + fabs(b_top));
  int64_t tf = t_top;
  if (tmax >= 0 && (tmax == t_top ? df_value(before) : mine) >= b_cut) {
    for (int64_t base = 0; base < t_top && tf == t_top; base += TILE)
      for (int64_t t = base + (int64_t)tid * K; t < min(base + (int64_t)(tid + 1) * K, t_top); ++t) {
        const double bd = boxcar(row, t);
        if (bd >= b_cut && (bd - mean) / sd == z_top) {
          tf = t;
          break;
        }
      }
  }
  tbest[tid] = tf;
  __syncthreads();
  for (int h = NT / 2; h > 0; h >>= 1) {
    if (tid < h) tbest[tid] = min(tbest[tid], tbest[tid + h]);
    __syncthreads();
  }
  if (tid == 0) put_stat(stats + i * stats_stride, RowStat{z_top, mean, sd, tbest[0]});
}

// One block: the best row (first on ties) -> result.
template <int NT>
__global__ void __launch_bounds__(NT) snr_pick_kernel(const float* __restrict__ stats, int64_t stride, int n_rows,
                                                      dd_snr_result* __restrict__ result) {
  __shared__ double zb[NT];
  __shared__ int ib[NT];
  double z = -DBL_MAX;
  int bi = -1;
  for (int i = threadIdx.x; i < n_rows; i += NT) {
    const RowStat r = get_stat(stats + i * stride);
    if (r.t >= 0 && r.z > z) {
      z = r.z;
      bi = i;
    }
  }
  zb[threadIdx.x] = z;
  ib[threadIdx.x] = bi;
  __syncthreads();
  for (int h = NT / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      const double zo = zb[threadIdx.x + h];
      const int io = ib[threadIdx.x + h];
      if (io >= 0 && (ib[threadIdx.x] < 0 || zo > zb[threadIdx.x] || (zo == zb[threadIdx.x] && io < ib[threadIdx.x]))) {
        zb[threadIdx.x] = zo;
        ib[threadIdx.x] = io;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    dd_snr_result r{};
    const int b = ib[0];
    if (b >= 0) {
      const RowStat best = get_stat(stats + b * stride);
      r.snr = best.z;
      r.loss = -best.z;
      r.mean = best.mean;
      r.std = best.sd;
      r.best_t = best.t;
      r.best_row = b;
      r.valid = 1;
    } else {
      r.best_row = -1;
      r.best_t = -1;
      r.valid = 0;
    }
    *result = r;
  }
}

// d loss / d x for the best row (the rows kernel cleared all).  Each boxcar and
// its double divisions eight times over made this one row cost 0.1 ms; every
// start's term is made once, with two divisions, and shared through the block.
template <int NT>
__global__ void __launch_bounds__(NT) snr_grad_kernel(const float* __restrict__ x, int64_t stride, int64_t n_cols,
                                                      const dd_snr_result* __restrict__ result, int n_rows,
                                                      float* __restrict__ grad, int64_t grad_stride) {
  // the other rows' statistics make place
  for (int64_t k = (int64_t)blockIdx.x * NT + threadIdx.x; k < (int64_t)n_rows * kBox; k += (int64_t)gridDim.x * NT)
    if (!result->valid || k / kBox != result->best_row) grad[k / kBox * grad_stride + k % kBox] = 0.0f;
  __shared__ double db[NT + kBox - 1];  // d snr / d b of the starts [u0 - 7, u0 + NT)
  if (!result->valid) return;
  const dd_snr_result r = *result;
  const int64_t u0 = (int64_t)blockIdx.x * NT;
  const float* row = x + (int64_t)r.best_row * stride;
  const int64_t nb = n_cols - kBox + 1;
  // d snr / d b[t] = ((t == best) - 1/nb) / sd - snr z[t] / (nb sd); divided, not
  // multiplied by reciprocals, so that two terms which cancel do so exactly
  const double inv_nb = 1.0 / (double)nb, nb_sd = (double)nb * r.std;
  const double at_best = (1.0 - inv_nb) / r.std, elsewhere = (0.0 - inv_nb) / r.std;
  for (int k = threadIdx.x; k < NT + kBox - 1; k += NT) {
    const int64_t t = u0 - (kBox - 1) + k;
    double v = 0.0;
    if (t >= 0 && t < nb) {
      const double z = (boxcar(row, t) - r.mean) / r.std;
      v = (t == r.best_t ? at_best : elsewhere) - r.snr * z / nb_sd;
    }
    db[k] = v;
  }
  __syncthreads();
  const int64_t u = u0 + threadIdx.x;
  if (u >= n_cols) return;
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < kBox; ++k) acc += db[threadIdx.x + k];
  grad[(int64_t)r.best_row * grad_stride + u] = (float)(-acc);
}

dd_status boxcar_snr_launch(const char* who, const float* x, int64_t row_stride, int32_t n_rows, int64_t n_cols,
                            dd_snr_result* result, float* grad, int64_t grad_stride, cudaStream_t s, void* scratch) {
  constexpr int NT = 256, K = 15;
  float* stats = grad ? grad : static_cast<float*>(scratch);
  const int64_t stats_stride = grad ? grad_stride : (int64_t)(sizeof(RowStat) / sizeof(float));
  if (grad)
    snr_rows_kernel<NT, K, true><<<n_rows, NT, 0, s>>>(x, row_stride, n_cols, stats, stats_stride, grad, grad_stride);
  else
    snr_rows_kernel<NT, K, false><<<n_rows, NT, 0, s>>>(x, row_stride, n_cols, stats, stats_stride, nullptr, 0);
  snr_pick_kernel<NT><<<1, NT, 0, s>>>(stats, stats_stride, n_rows, result);
  if (grad)
    snr_grad_kernel<NT><<<(unsigned)((n_cols + NT - 1) / NT), NT, 0, s>>>(x, row_stride, n_cols, result, n_rows, grad,
                                                                          grad_stride);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return set_error(DD_ERR_CUDA, "%s: launch: %s (%s)", who, cudaGetErrorString(e),
                                         cudaGetErrorName(e));
  return DD_OK;
}

dd_status boxcar_snr_check(const char* who, const float* x, int64_t row_stride, int32_t n_rows, int64_t n_cols,
                           const dd_snr_result* result, const float* grad, int64_t grad_stride) {
  if (!x || !result) return set_error(DD_ERR_ARG, "%s: x/result is NULL", who);
  if (n_rows <= 0) return set_error(DD_ERR_ARG, "%s: n_rows must be > 0", who);
  if (n_cols < kBox) return set_error(DD_ERR_SHAPE, "%s: n_cols must be >= %d", who, kBox);
  if (row_stride < n_cols) return set_error(DD_ERR_SHAPE, "%s: row_stride < n_cols", who);
  if (grad && grad_stride < n_cols) return set_error(DD_ERR_SHAPE, "%s: grad_stride < n_cols", who);
  return DD_OK;
}

}  // namespace dd

using namespace dd;

extern "C" dd_status dd_boxcar_snr(const float* x, int64_t row_stride, int32_t n_rows, int64_t n_cols,
                                   dd_snr_result* result, float* grad, int64_t grad_stride, void* stream) {
  NvtxRange range("dd_boxcar_snr");
  clear_error();
  dd_status st = boxcar_snr_check("dd_boxcar_snr", x, row_stride, n_rows, n_cols, result, grad, grad_stride);
  if (st != DD_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // The allocator gives memory back at every synchronisation and then takes
  // 0.2 ms to get it again, as long as the rest of the call.
  if (grad)
    return boxcar_snr_launch("dd_boxcar_snr", x, row_stride, n_rows, n_cols, result, grad, grad_stride, s, nullptr);
  void* scratch = nullptr;
  const size_t bytes = (size_t)n_rows * sizeof(RowStat);
  if (cudaMallocAsync(&scratch, bytes, s) != cudaSuccess)
    return set_error(DD_ERR_NOMEM, "dd_boxcar_snr: cannot allocate %zu bytes of scratch", bytes);
  st = boxcar_snr_launch("dd_boxcar_snr", x, row_stride, n_rows, n_cols, result, grad, grad_stride, s, scratch);
  cudaFreeAsync(scratch, s);
  return st;
}

// ------------------------------------------------------ allocation-free form
// Per-row scratch for dd_boxcar_snr_noalloc without a gradient (with one, the
// statistics wait in its rows).  It is part of the library image,
// so each GPU that loads the library carries it (2 MiB) until the process
// exits, and no call ever has to allocate.  Host code cannot use the symbol
// itself as a device address: the address is looked up per device below.
namespace dd {
static __device__ __align__(256) RowStat g_noalloc_rows[DD_NOALLOC_MAX_ROWS];
constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
// per device: the context the address was looked up in, and the address
struct NoAllocSlot {
  void* ctx = nullptr;
  void* addr = nullptr;
};
static NoAllocSlot g_noalloc[kNoAllocMaxDevices];

typedef int (*CtxGetCurrentFn)(void**);
// The driver's cuCtxGetCurrent, looked up once through the runtime.
static CtxGetCurrentFn ctx_get_current() {
  static CtxGetCurrentFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<CtxGetCurrentFn>(p);
  });
  return fn;
}

// Device address of g_noalloc_rows on the current device, looked up on the
// first call for that device, and again whenever the device's context has
// changed since (after cudaDeviceReset the array lives in the new context).
static dd_status noalloc_rows(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_cuda_error("dd_boxcar_snr_noalloc: cudaGetDevice", e);
  if (dev < 0 || dev >= kNoAllocMaxDevices)
    return set_error(DD_ERR_UNSUPPORTED, "dd_boxcar_snr_noalloc: device %d is beyond the %d supported", dev,
                     kNoAllocMaxDevices);
  // make sure the device's primary context exists and is current
  e = cudaFree(nullptr);
  if (e != cudaSuccess) return set_cuda_error("dd_boxcar_snr_noalloc: context", e);
  void* ctx = nullptr;
  CtxGetCurrentFn get = ctx_get_current();
  if (!get || get(&ctx) != 0 || !ctx)
    return set_error(DD_ERR_CUDA, "dd_boxcar_snr_noalloc: cannot read the current context");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  NoAllocSlot& slot = g_noalloc[dev];
  if (!slot.addr || slot.ctx != ctx) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_rows);
    if (e != cudaSuccess || !p) return set_cuda_error("dd_boxcar_snr_noalloc: cudaGetSymbolAddress", e);
    slot.ctx = ctx;
    slot.addr = p;
  }
  *out = slot.addr;
  return DD_OK;
}
}  // namespace dd

extern "C" dd_status dd_boxcar_snr_noalloc(const float* x, int64_t row_stride, int32_t n_rows, int64_t n_cols,
                                           dd_snr_result* result, float* grad, int64_t grad_stride, void* stream) {
  NvtxRange range("dd_boxcar_snr_noalloc");
  clear_error();
  dd_status st = boxcar_snr_check("dd_boxcar_snr_noalloc", x, row_stride, n_rows, n_cols, result, grad, grad_stride);
  if (st != DD_OK) return st;
  if (n_rows > DD_NOALLOC_MAX_ROWS)
    return set_error(DD_ERR_SHAPE, "dd_boxcar_snr_noalloc: %d rows exceed the fixed scratch of %d rows", n_rows,
                     DD_NOALLOC_MAX_ROWS);
  void* rows = nullptr;
  st = noalloc_rows(&rows);
  if (st != DD_OK) return st;
  return boxcar_snr_launch("dd_boxcar_snr_noalloc", x, row_stride, n_rows, n_cols, result, grad, grad_stride,
                           static_cast<cudaStream_t>(stream), rows);
}
