"""The weight gradient when few rows of grad_out have a nonzero: the listed
rows alone (up to 8, and at most half), the tiles past that, and the tiles
again where the input holds an infinity, whose product with a zero is not zero."""
import numpy as np
import pytest

import oracle
from paper_1601_01165_gb300 import synth
from helpers import FP32_REL, make_input, oracle_table

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(dd, n_dm, n_out, rows, seed=5):
    s = synth.Setup("few", 130, 1420.0, 2.0, 50e-6, 0.0, 0.25, n_dm, n_out)
    plan = dd.Plan.from_setup(s, "f32")
    assert "tmw9_f32_d9_t4096" in plan.configs()
    d = oracle_table(s)
    x, _ = make_input(s, "f32", seed, plan.n_in, plan.padded_in_stride())
    x[:, plan.n_in:] = np.nan                       # row padding never counts
    g = np.zeros((n_dm, n_out), dtype=np.float32)
    g[rows] = synth.noise_f32(seed + 1, n_dm, n_out)[rows]
    return plan, d, x, g


@pytest.mark.parametrize("n_dm,rows", [(40, []), (40, [0]), (40, [39]), (40, [3, 4, 5, 17, 20, 21, 22, 38]),
                                       (40, list(range(9))), (3, [0, 2]), (1, [0]), (1500, [700, 1499])])
@pytest.mark.parametrize("n_out", [255, 3001])
def test_few_rows_match_oracle(n_dm, rows, n_out):
    from paper_1601_01165_gb300 import binding as dd
    plan, d, x, g = _case(dd, n_dm, n_out, rows)
    xt, gt = torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda()
    _, gw = plan.adjoint(gt, x=xt, grad_in=False, grad_w=True)
    _, again = plan.adjoint(gt, x=xt, grad_in=False, grad_w=True)
    assert plan.device_status() == 0 and torch.equal(gw, again)
    xs = np.ascontiguousarray(x[:, :plan.n_in])
    ref, scale = oracle.wgrad_f32(d, g, xs), oracle.wgrad_f32(d, np.abs(g), np.abs(xs))
    assert (np.abs(gw.cpu().numpy().astype(np.float64) - ref) <= FP32_REL * scale).all()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_sample_that_is_not_finite_counts_in_zero_rows(bad):
    from paper_1601_01165_gb300 import binding as dd
    plan, d, x, g = _case(dd, 40, 3001, [7])
    x[5, 1000] = bad
    _, gw = plan.adjoint(torch.from_numpy(g).cuda(), x=torch.from_numpy(x).cuda(), grad_in=False, grad_w=True)
    got = gw.cpu().numpy()
    assert np.isnan(got[5]) and np.isfinite(np.delete(got, 5)).all()
