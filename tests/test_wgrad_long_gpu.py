"""The few-row weight gradient of a long row.  Every product is 1 + 0.45 * 2^-13,
whose fraction a float sum past 1024 drops (the rounding unit there is 2^-13):
sums that grow with the row's length lose 2e-5 of it, sums of a fixed number of
products do not."""
import numpy as np
import pytest

from paper_1601_01165_gb300 import synth
from helpers import FP32_REL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [[4], [0, 3, 8]])
@pytest.mark.parametrize("n_out", [200_003, 2_000_000])
def test_long_rows_keep_their_precision(n_out, rows):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("long", 8, 1420.0, 300.0 / 8, 50e-6, 0.0, 0.25, 9, n_out)
    plan = dd.Plan.from_setup(s, "f32")
    assert "tmw9_f32_d9_t4096" in plan.configs()
    x = plan.alloc_input()
    x[:, :plan.n_in] = 1.0
    g = torch.zeros((s.n_dm, n_out), device="cuda")
    p = np.float32(1.0 + 0.45 * 2.0 ** -13)
    g[rows] = float(p)
    _, gw = plan.adjoint(g, x=x, grad_in=False, grad_w=True)
    assert plan.device_status() == 0
    want = len(rows) * n_out * float(p)
    # chains of 16 products round 16 times by half a unit at most, the result once
    assert 17 * 2.0 ** -24 < FP32_REL
    assert (np.abs(gw.cpu().numpy().astype(np.float64) - want) <= 17 * 2.0 ** -24 * want).all()
