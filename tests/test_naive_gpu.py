"""The plain kernel around its batches of channels (16 float, 32 uint8): fewer
channels than one, one more or less, and a remainder after several."""
import numpy as np
import pytest

from paper_1601_01165_gb300 import synth
from helpers import assert_parity, make_input, oracle_table, oracle_window

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 97])
@pytest.mark.parametrize("dtype,weighted", [("f32", False), ("f32", True), ("u8", False)])
def test_channel_counts_around_a_batch(C, dtype, weighted):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("naive", C, 1420.0, 300.0 / C, 50e-6, 2.0, 0.5, 7, 300)
    plan = dd.Plan.from_setup(s, dtype)
    d = oracle_table(s)
    x, _ = make_input(s, dtype, C, plan.n_in + 1)
    w = synth.weights(C, C) if weighted else None
    ref, scale = oracle_window(d, x, dtype, 0, s.n_dm, 0, s.n_out, w)
    xt = torch.from_numpy(x).cuda()
    wt = torch.from_numpy(np.ascontiguousarray(w)).cuda() if weighted else None
    for cfg in plan.configs():
        if cfg.startswith("naive"):
            plan.select(cfg)
            got = plan.forward(xt, wt)
            assert_parity(got.cpu().numpy(), ref, scale, dtype, where=f"{C} {dtype} {cfg}")
