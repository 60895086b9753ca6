"""Runs adjoints and weight gradients of every route through the library named
by DD_LIBRARY (the checked build, whose kernels record any out-of-range index in
the plan's status word instead of making the access) and compares with the
oracle.  Exits nonzero on the first problem.  Started by
tests/test_checked_adjoint_gpu.py in a process of its own."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import torch  # noqa: E402

import oracle  # noqa: E402
from paper_1601_01165_gb300 import binding as dd, synth  # noqa: E402
from helpers import FP32_REL, make_input, oracle_table  # noqa: E402


def _apertif(C, n_dm, n_out, step=0.25):
    return synth.Setup(f"{C}x{n_dm}x{n_out}", C, 1420.0, 300.0 / C, 50e-6, 0.0, step, n_dm, n_out)


SETUPS = [
    # (the transposed plans of the first three choose float grouped sums; the host-path tests see to it)
    _apertif(1024, 70, 9001), _apertif(700, 64, 9000), _apertif(1019, 33, 12345),
    _apertif(130, 40, 3001), _apertif(37, 3, 1001), _apertif(33, 25, 2999, 16.0),
    synth.Setup("lofar-cut", 32, 138.0, 0.1953125, 5e-6, 0.0, 0.01, 70, 3001),
]


def main():
    dd.load()
    assert "checked" in os.environ.get("DD_LIBRARY", ""), "run with DD_LIBRARY naming the checked build"
    for s in SETUPS:
        d = oracle_table(s)
        plan = dd.Plan.from_setup(s, "f32")
        x, _ = make_input(s, "f32", 3, plan.n_in, plan.padded_in_stride())
        xs = np.ascontiguousarray(x[:, :plan.n_in])
        xt, w = torch.from_numpy(x).cuda(), synth.weights(4, s.channels)
        wt = torch.from_numpy(w).cuda()
        dense = synth.noise_f32(5, s.n_dm, s.n_out)
        few = np.zeros_like(dense)
        few[s.n_dm // 2] = dense[s.n_dm // 2]
        for name, g, grad_in, grad_w in (("grad_in", dense, True, False), ("both", dense, True, True),
                                         ("grad_w", dense, False, True), ("grad_w of one row", few, False, True)):
            gi, gw = plan.adjoint(torch.from_numpy(g).cuda(), w=wt, x=xt, grad_in=grad_in, grad_w=grad_w)
            torch.cuda.synchronize()
            code = plan.device_status()
            if code != 0:
                print(f"{s.name} {name}: device status {code}")
                return 1
            if gi is not None:
                ref = oracle.adjoint_f32(d, g, plan.n_in, w)
                lim = FP32_REL * oracle.adjoint_f32(d, np.abs(g), plan.n_in, np.abs(w))
                assert (np.abs(gi.cpu().numpy() - ref) <= lim).all(), (s.name, name, "grad_in")
            if gw is not None:
                ref, lim = oracle.wgrad_f32(d, g, xs), FP32_REL * oracle.wgrad_f32(d, np.abs(g), np.abs(xs))
                assert (np.abs(gw.cpu().numpy() - ref) <= lim).all(), (s.name, name, "grad_w")
    print("checked build: adjoints in range and equal to the oracle")
    return 0


if __name__ == "__main__":
    sys.exit(main())
