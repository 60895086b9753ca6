"""Which kernels the library's host code launches, and what it does when memory
runs out, without a GPU: the library's own objects linked with a CUDA runtime
that only records launches (fake_cudart.cpp)."""
import ctypes
import glob
import json
import os
import subprocess

import pytest

from paper_1601_01165_gb300 import build, synth

HERE = os.path.dirname(os.path.abspath(__file__))
U8, F32 = 0, 1


class Host:
    """The library on the recording runtime."""

    def __init__(self, path):
        lib = self.lib = ctypes.CDLL(path)
        i32, i64, dbl, vp = ctypes.c_int32, ctypes.c_int64, ctypes.c_double, ctypes.c_void_p
        lib.dd_plan.argtypes = [ctypes.POINTER(vp), i32, dbl, dbl, dbl, dbl, dbl, i32, i64, ctypes.c_int]
        lib.dd_plan_config_name.argtypes, lib.dd_plan_config_name.restype = [vp, i32], ctypes.c_char_p
        lib.dd_plan_select_config.argtypes = [vp, i32]
        lib.dd_plan_selected_config.argtypes = [vp, ctypes.POINTER(i32)]
        lib.dd_plan_num_configs.argtypes = [vp, ctypes.POINTER(i32)]
        lib.dd_plan_destroy.argtypes = [vp]
        lib.dd_tune.argtypes = [vp, dbl, ctypes.c_char_p, ctypes.POINTER(dbl)]
        lib.dd_forward.argtypes = [vp, vp, i64, vp, vp, i64, vp]
        lib.dd_plan_in_stride.argtypes = [vp, ctypes.POINTER(i64)]
        lib.dd_stream_create.argtypes = [ctypes.POINTER(vp), vp, i64]
        lib.dd_stream_push.argtypes = [vp, vp, vp, ctypes.POINTER(i64), vp]
        lib.dd_stream_destroy.argtypes = [vp]
        lib.fake_launch_name.restype = ctypes.c_char_p

    def plan(self, setup, dtype):
        h = ctypes.c_void_p()
        assert self.lib.dd_plan(ctypes.byref(h), *setup.plan_args(), dtype) == 0
        return h

    def configs(self, h):
        n = ctypes.c_int32()
        self.lib.dd_plan_num_configs(h, ctypes.byref(n))
        return [self.lib.dd_plan_config_name(h, k).decode() for k in range(n.value)]

    def selected(self, h):
        k = ctypes.c_int32()
        self.lib.dd_plan_selected_config(h, ctypes.byref(k))
        return self.configs(h)[k.value]

    def launches(self, call):
        self.lib.fake_clear_launches()
        assert call() == 0
        return [self.lib.fake_launch_name(k).decode() for k in range(self.lib.fake_launches())]

    def forward(self, h):
        stride = ctypes.c_int64()
        self.lib.dd_plan_in_stride(h, ctypes.byref(stride))
        return self.launches(lambda: self.lib.dd_forward(h, 4096, stride.value, None, 8192, 1 << 30, None))

    def push(self, h, chunk):
        """The kernels one push into a stream made from the plan launches."""
        st, t0 = ctypes.c_void_p(), ctypes.c_int64()
        assert self.lib.dd_stream_create(ctypes.byref(st), h, chunk) == 0
        names = self.launches(lambda: self.lib.dd_stream_push(st, 4096, 8192, ctypes.byref(t0), None))
        self.lib.dd_stream_destroy(st)
        return names


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    build.build()
    out = str(tmp_path_factory.mktemp("host") / "libdd_host.so")
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-o", out, os.path.join(HERE, "fake_cudart.cpp"), *objs,
                    "-Wl,--no-undefined", "-Wl,-Bsymbolic", "-lpthread", "-ldl"], check=True)
    return Host(out)


def _apertif(n_out, n_dm=2048, C=1024):
    return synth.Setup("host", C, 1420.0, 300.0 / C, 50e-6, 0.0, 0.25, n_dm, n_out)


# ------------------------------------------------------------------ streams
@pytest.mark.parametrize("dtype", [F32, U8], ids=["f32", "u8"])
@pytest.mark.parametrize("n_dm", [64, 512])
@pytest.mark.parametrize("chunk", [500, 20000])
def test_a_stream_chooses_for_its_chunks(host, dtype, n_dm, chunk):
    """Whatever the plan's n_out: a push runs the kernel that a forward call of the chunk's length would."""
    want = host.forward(host.plan(_apertif(chunk, n_dm), dtype))
    for n_out in (1, 256, 1000, 20000):
        assert host.push(host.plan(_apertif(n_out, n_dm), dtype), chunk) == want, n_out


@pytest.mark.parametrize("dtype", [F32, U8], ids=["f32", "u8"])
def test_a_stream_keeps_what_was_selected(host, dtype):
    for name in host.configs(host.plan(_apertif(1, 64), dtype)):
        chunk_plan = host.plan(_apertif(3000, 64), dtype)
        host.lib.dd_plan_select_config(chunk_plan, host.configs(chunk_plan).index(name))
        want = host.forward(chunk_plan)
        h = host.plan(_apertif(1, 64), dtype)
        host.lib.dd_plan_select_config(h, host.configs(h).index(name))
        assert host.push(h, 3000) == want, name
    h = host.plan(_apertif(1, 64), dtype)
    assert host.lib.dd_tune(h, 0.0, None, None) == 0     # every time the same here: the most promising one
    name = host.selected(h)
    chunk_plan = host.plan(_apertif(3000, 64), dtype)
    host.lib.dd_plan_select_config(chunk_plan, host.configs(chunk_plan).index(name))
    assert host.push(h, 3000) == host.forward(chunk_plan)


def test_a_stream_and_the_tuning_database(host, tmp_path, monkeypatch):
    """An entry for the plan holds for its streams, unless there is one for the chunks' own length; a selection wins."""
    def key(n_out):
        s = _apertif(n_out, 64)
        return (f"fake|C={s.channels}|f_low=1420|chan_bw={s.chan_bw_mhz:.9g}|t_samp=5e-05|dm_first=0|dm_step=0.25|"
                f"n_dm=64|n_out={n_out}|f32")

    def entry(n_out, name):
        return json.dumps({"key": key(n_out), "config": name, "ms": 1.0}) + "\n"

    db = tmp_path / "tune.jsonl"
    monkeypatch.setenv("DD_TUNE_DB", str(db))

    def kernel(name):
        h = host.plan(_apertif(777, 64), F32)
        host.lib.dd_plan_select_config(h, host.configs(h).index(name))
        return host.forward(h)

    db.write_text(entry(1000, "staged_d64_t256_c4_s3"))
    h = host.plan(_apertif(1000, 64), F32)
    assert host.selected(h) == "staged_d64_t256_c4_s3"
    assert host.push(h, 3000) == kernel("staged_d64_t256_c4_s3")
    db.write_text(entry(1000, "staged_d64_t256_c4_s3") + entry(3000, "naive_t32"))
    h = host.plan(_apertif(1000, 64), F32)
    assert host.push(h, 3000) == kernel("naive_t32")
    host.lib.dd_plan_select_config(h, host.configs(h).index("staged_d16_t256_c8_s3"))
    assert host.push(h, 3000) == kernel("staged_d16_t256_c8_s3")


# ------------------------------------------------------- choice on steep grids
# (band, channels, trials, samples, DM step; the configurations within 15 % of
# the fastest of the menu as timed on the GPU, fastest first)
STEEP = [
    ("lofar", 30, 477, 66978, 0.32, U8, ["staged_d8_t1024_c4_s3"]),                       # 161 us; plain 445
    ("lofar", 18, 242, 81259, 0.32, U8, ["staged_d8_t1024_c4_s3"]),                       # 66; 181
    ("apertif", 521, 257, 17780, 16.0, U8, ["u8pk_w4x2_d2_c16_st4", "u8pk_w8x2_d1_c16_st4"]),  # 244; 811
    ("apertif", 389, 179, 41677, 64.0, U8, ["staged_d8_t1024_c4_s3"]),                    # 535; 991
    ("lofar", 23, 1455, 25939, 0.01, U8, ["u8pk_w8x1_d2_c16_st4"]),                       # 76; 32-channel chunks 103
    ("apertif", 447, 223, 17992, 8.0, F32, ["staged_d8_t1024_c4_s3"]),                    # 325; d8 t512 553
    ("lofar", 229, 458, 16729, 0.04, F32, ["staged_d8_t1024_c4_s3"]),                     # 309; d8 t512 529
    ("apertif", 52, 3471, 8917, 4.0, F32, ["staged_d8_t1024_c4_s3"]),                     # 212; d32 t512 277
    ("lofar", 766, 6, 2812, 0.64, U8, ["naive_t128"]),                                    # 19; staged 238
    ("lofar", 449, 55, 2424, 0.02, F32, ["naive_t128"]),                                  # 29; staged 140
]


@pytest.mark.parametrize("band,C,n_dm,n_out,step,dtype,good", STEEP)
def test_default_on_steep_grids(host, band, C, n_dm, n_out, step, dtype, good):
    f_low, bw, t_samp = {"apertif": (1420.0, 300.0, 50e-6), "lofar": (138.0, 6.25, 5e-6)}[band]
    assert host.selected(host.plan(synth.Setup("steep", C, f_low, bw / C, t_samp, 0.0, step, n_dm, n_out), dtype)) in good


@pytest.mark.parametrize("C,n_dm,n_out,step", [(460, 641, 18008, 0.25), (753, 118, 21229, 2.0)])
def test_adjoint_too_steep_for_nine_trials_takes_six(host, C, n_dm, n_out, step):
    """705 and 244 us with six-trial windows; staged 841 and 279."""
    i64, vp = ctypes.c_int64, ctypes.c_void_p
    host.lib.dd_adjoint.argtypes = [vp, vp, i64, vp, vp, i64, vp, i64, vp, vp]
    h = host.plan(synth.Setup("steep", C, 1420.0, 300.0 / C, 50e-6, 0.0, step, n_dm, n_out), F32)
    names = host.launches(lambda: host.lib.dd_adjoint(h, 4096, 1 << 40, None, 8192, 1 << 40, None, 0, None, None))
    assert len(names) == 1 and "fwd_tmw6_kernel" in names[0], names


# ------------------------------------------------------------------- memory
@pytest.mark.parametrize("C,n_dm", [(192, 1), (193, 3), (250, 64), (1000, 65), (1024, 255), (1024, 512), (700, 130)])
def test_footprint_is_what_a_plan_holds(host, C, n_dm):
    """With the grouped-sum tables of every shape the plan offers."""
    i32, i64, dbl = ctypes.c_int32, ctypes.c_int64, ctypes.c_double
    s = _apertif(3000, n_dm, C)
    host.lib.dd_plan_footprint.argtypes = [i32, dbl, dbl, dbl, dbl, dbl, i32, ctypes.c_int, ctypes.POINTER(i64)]
    host.lib.dd_plan_info.argtypes = [ctypes.c_void_p, ctypes.POINTER(i64), ctypes.POINTER(i32), ctypes.POINTER(i64)]
    sized, held = i64(), i64()
    assert host.lib.dd_plan_footprint(*s.plan_args()[:7], U8, ctypes.byref(sized)) == 0
    h = host.plan(s, U8)
    assert C < 1000 or any(c.startswith("gsum8") for c in host.configs(h))
    host.lib.dd_plan_info(h, None, None, ctypes.byref(held))
    assert sized.value == held.value


@pytest.mark.parametrize("n_dm", [64, 600])
def test_a_plan_without_room_for_grouped_sums_works_without_them(host, n_dm):
    """Allocations failing one after another: the delay tables are needed, the
    grouped-sum tables are not.  Nothing is left behind either way."""
    i32, i64 = ctypes.c_int32, ctypes.c_int64
    host.lib.dd_plan_info.argtypes = [ctypes.c_void_p, ctypes.POINTER(i64), ctypes.POINTER(i32), ctypes.POINTER(i64)]
    host.lib.fake_fail_malloc.argtypes = [ctypes.c_long]
    host.lib.fake_live.restype = ctypes.c_long
    s = _apertif(20000, n_dm)
    live = host.lib.fake_live()

    def make(fail):
        host.lib.fake_fail_malloc(fail)
        h, held = ctypes.c_void_p(), i64()
        status = host.lib.dd_plan(ctypes.byref(h), *s.plan_args(), U8)
        host.lib.fake_fail_malloc(0)
        if status != 0:
            assert host.lib.fake_live() == live
            return status, None, None, None
        names, chosen = host.configs(h), host.selected(h)
        host.lib.dd_plan_info(h, None, None, ctypes.byref(held))
        assert len(host.forward(h)) == 1
        host.lib.dd_plan_destroy(h)
        assert host.lib.fake_live() == live
        return 0, names, chosen, held.value

    status, names, chosen, held = make(0)
    shapes = [c for c in names if c.startswith("gsum8")]
    assert status == 0 and chosen in shapes
    for k in (1, 2, 3):                                  # delays, their transpose, the status word
        assert make(k)[0] == 4, k                        # DD_ERR_NOMEM
    for k in range(4, 4 + 2 * len(shapes)):              # two tables a shape
        status, left, chosen_now, held_now = make(k)
        missing = shapes[(k - 4) // 2]
        assert status == 0, k
        assert left == [c for c in names if c != missing] and chosen_now in left and held_now < held
    assert make(4 + 2 * len(shapes)) == (0, names, chosen, held)


def test_the_adjoint_uses_shared_sums_where_it_is_tested(host):
    """The sizes by which tests/test_gsum_gpu.py means to run float GSUM do."""
    i64, vp = ctypes.c_int64, ctypes.c_void_p
    host.lib.dd_adjoint.argtypes = [vp, vp, i64, vp, vp, i64, vp, i64, vp, vp]
    for C, n_dm, n_out in [(1024, 70, 9001), (700, 64, 9000), (1019, 33, 12345), (1024, 2048, 20000)]:
        h = host.plan(_apertif(n_out, n_dm, C), F32)
        names = host.launches(lambda: host.lib.dd_adjoint(h, 4096, 1 << 40, None, 8192, 1 << 40, None, 0, None, None))
        assert len(names) == 1 and "fwd_gsum_kernelIf" in names[0], (C, n_dm, n_out, names)
