"""GSUM (sums of eight channels made once per delay pattern) at its edges:
channel counts that leave a last group of 1..7, trial counts around its blocks,
time tails around its tiles, more than 256 channels (its packed 8-bit sums are
emptied every 32 groups), first trials past zero, saturated samples; and, on
float, the adjoint's transposed plan, whose delays grow with the channel."""
import numpy as np
import pytest

import oracle
from paper_1601_01165_gb300 import synth
from helpers import FP32_REL, assert_parity, make_input, oracle_table, oracle_window

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gsum(plan):
    return [c for c in plan.configs() if c.startswith("gsum8")]


@pytest.mark.parametrize("C,n_dm,n_out,dm0", [
    (193, 1, 1, 0.0), (199, 15, 447, 0.0), (200, 17, 448, 0.0), (250, 33, 449, 300.0), (257, 64, 1345, 0.0),
    (515, 65, 900, 40.0), (1024, 31, 1931, 400.0), (1022, 130, 463, 0.0), (1024, 70, 577, 0.0), (777, 64, 1151, 200.0),
])
@pytest.mark.parametrize("saturated", [False, True], ids=["noise", "saturated"])
def test_u8_every_shape_is_exact(C, n_dm, n_out, dm0, saturated):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("gsum", C, 1420.0, 0.29296875, 50e-6, dm0, 0.25, n_dm, n_out)
    plan = dd.Plan.from_setup(s, "u8")
    names = _gsum(plan)
    assert names, "this grid's patterns are few enough"
    d = oracle_table(s)
    x, _ = make_input(s, "u8", C + n_dm, plan.n_in, plan.padded_in_stride())
    if saturated:
        x[:, :plan.n_in] = np.where(x[:, :plan.n_in] > 110, 255, 0)
    ref, _ = oracle_window(d, x, "u8", 0, n_dm, 0, n_out)
    xt = torch.from_numpy(x).cuda()
    for cfg in names:
        plan.select(cfg)
        big = torch.full((n_dm, n_out + 3), -7, dtype=torch.int32, device="cuda")
        plan.forward(xt, out=big[:, :n_out])
        assert plan.device_status() == 0, cfg
        got = big.cpu().numpy()
        assert (got[:, n_out:] == -7).all()
        assert_parity(got[:, :n_out], ref, None, "u8", where=f"{s} {cfg}")


# (sizes at which GSUM is the transposed plan's choice; 70, 64, 33 "channels" there)
@pytest.mark.parametrize("C,n_dm,n_out", [(1024, 70, 9001), (700, 64, 9000), (1019, 33, 12345)])
def test_adjoint_on_the_transposed_plan(C, n_dm, n_out):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("gsum-adj", C, 1420.0, 300.0 / C, 50e-6, 0.0, 0.25, n_dm, n_out)
    plan = dd.Plan.from_setup(s, "f32")
    assert not _gsum(plan)                          # float forwards add channel by channel
    d = oracle_table(s)
    g, w = synth.noise_f32(8, n_dm, n_out), synth.weights(8, C)
    gi, _ = plan.adjoint(torch.from_numpy(g).cuda(), w=torch.from_numpy(w).cuda())
    assert plan.device_status() == 0
    ref, scale = oracle.adjoint_f32(d, g, plan.n_in, w), oracle.adjoint_f32(d, np.abs(g), plan.n_in, np.abs(w))
    assert (np.abs(gi.cpu().numpy().astype(np.float64) - ref) <= FP32_REL * scale).all()
