"""Copies of input rows that start anywhere (spans.h), compiled for the host:
they cover what a tile needs, on 16-byte boundaries, and read nothing after the
last sample of the last row, which may be the last of the caller's memory."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_01165_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "spans.h"
template <int V>
static int check() {
  for (int64_t n_in = 40; n_in < 40 + 2 * V; ++n_in)
    for (int64_t stride = n_in; stride < n_in + 2 * V + 3; ++stride)
      for (int C = 1; C <= 3; ++C)
        for (int c = 0; c < C; ++c)
          for (int64_t from = 0; from < n_in; ++from)
            for (int64_t to = from + 1; to <= n_in; ++to) {
              const int64_t row = c * stride, end = dd::input_end(C, stride, n_in);
              const dd::RowSpan s = dd::row_span<V>(row + from, row + to, end);
              const bool ok = s.first >= 0 && s.first % V == 0 && s.bulk_end % V == 0 && s.first <= row + from &&
                              row + from - s.first < V && s.first <= s.bulk_end && s.bulk_end <= s.last &&
                              s.last >= row + to && s.last <= (C - 1) * stride + n_in && s.last - s.bulk_end < V &&
                              s.last - s.first <= to - from + 2 * V - 2;
              if (!ok) {
                std::printf("V %d n_in %ld stride %ld C %d c %d from %ld to %ld: %ld %ld %ld\n", V, (long)n_in,
                            (long)stride, C, c, (long)from, (long)to, (long)s.first, (long)s.bulk_end, (long)s.last);
                return 1;
              }
            }
  return 0;
}
int main() { return check<4>() || check<16>(); }
"""


def test_spans_cover_and_stay_inside(tmp_path):
    src, exe = tmp_path / "spans.cpp", tmp_path / "spans"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_the_kernels_use_them():
    # the copies of rows that start anywhere take their bounds from these functions
    with open(os.path.join(CSRC, "fwd_kernels.cu")) as f:
        text = f.read()
    assert "input_end(a.C, a.in_stride, a.n_in)" in text and "row_span<V>(" in text
