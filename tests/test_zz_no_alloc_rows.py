"""dd_boxcar_snr_noalloc without a gradient: the only calls that keep their row
statistics in the library's fixed array (with one, the statistics wait in the
gradient's rows)."""
import ctypes
import struct

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAX_ROWS = 65536  # DD_NOALLOC_MAX_ROWS in include/dd.h


@pytest.fixture(scope="module")
def call():
    from paper_1601_01165_gb300 import binding
    lib = binding.load()
    vp, i32, i64 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64

    def run(name, x, grad=False):
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = ctypes.c_int, [vp, i64, i32, i64, vp, vp, i64, vp]
        res = torch.zeros(48, dtype=torch.uint8, device="cuda")
        g = torch.empty_like(x) if grad else None
        rc = fn(x.data_ptr(), x.stride(0), x.shape[0], x.shape[1], res.data_ptr(), g.data_ptr() if grad else None,
                g.stride(0) if grad else 0, torch.cuda.current_stream().cuda_stream)
        assert rc == 0, lib.dd_last_error()
        return struct.unpack("<4dqii", bytes(res.cpu().numpy().tobytes()))

    return run


def _block(seed, rows, cols, best_row):
    x = torch.randn((rows, cols), generator=torch.Generator(device="cpu").manual_seed(seed))
    x[best_row, cols // 2: cols // 2 + 5] += 9.0
    return x.cuda()


def test_statistics_in_the_fixed_array_are_the_others(call):
    # a larger block first: what it leaves in the array must not count for the smaller ones
    for seed, rows, cols, best in ((1, 5000, 700, 4999), (2, 300, 2000, 100), (3, 1, 64, 0), (4, 517, 1333, 0)):
        x = _block(seed, rows, cols, best)
        want = call("dd_boxcar_snr", x)
        assert call("dd_boxcar_snr_noalloc", x) == want and want[5] == best and want[6] == 1
        assert call("dd_boxcar_snr_noalloc", x, grad=True) == want == call("dd_boxcar_snr", x, grad=True)


def test_rows_without_a_deviation_leave_the_array_invalid(call):
    call("dd_boxcar_snr_noalloc", _block(5, 40, 100, 7))
    assert call("dd_boxcar_snr_noalloc", torch.full((40, 100), 0.5, device="cuda"))[5:] == (-1, 0)


def test_the_arrays_last_entry(call):
    x = _block(6, MAX_ROWS, 256, MAX_ROWS - 1)
    got = call("dd_boxcar_snr_noalloc", x)
    assert got == call("dd_boxcar_snr", x) and got[5] == MAX_ROWS - 1 and got[6] == 1
