// Where the copies of input spans begin and end, for rows that start anywhere.
// Plain arithmetic without CUDA, so that it can be checked on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define DD_HOST_DEVICE inline
#endif

namespace dd {

// Samples are counted from the input's first one, rows of in_stride samples.
// The caller's rows may be a part of wider ones, so the last row is known to be
// there only as far as a launch reads it: n_in samples.
DD_HOST_DEVICE int64_t input_end(int32_t C, int64_t in_stride, int64_t n_in) {
  return (int64_t)(C - 1) * in_stride + n_in;
}

// The samples [from, to) of an input, widened to whole 16-byte groups of V
// samples: a bulk copy takes [first, bulk_end), and [bulk_end, last) is copied
// one by one (bulk_end < last only where the groups would pass `end`).
struct RowSpan {
  int64_t first, bulk_end, last;
};
template <int V>
DD_HOST_DEVICE RowSpan row_span(int64_t from, int64_t to, int64_t end) {
  static_assert((V & (V - 1)) == 0, "a power of two");
  RowSpan s;
  s.first = from & ~(int64_t)(V - 1);
  s.last = s.bulk_end = (to + V - 1) & ~(int64_t)(V - 1);
  if (s.last > end) {
    s.last = end;
    s.bulk_end = end & ~(int64_t)(V - 1);
  }
  return s;
}

}  // namespace dd
