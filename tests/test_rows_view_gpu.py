"""Input rows that are a part of wider ones: a view whose last row ends with
the tensor's memory, in strides that start rows anywhere."""
import pytest

from paper_1601_01165_gb300 import synth
from helpers import assert_parity, make_input, oracle_table, oracle_window

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,off", [("f32", 4), ("f32", 12), ("u8", 16), ("u8", 48)])
@pytest.mark.parametrize("C,n_dm,n_out,step", [(33, 9, 1001, 0.25), (40, 20, 2998, 0.0), (64, 70, 1503, 0.25)])
def test_a_view_that_ends_with_its_tensor(dtype, off, C, n_dm, n_out, step):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("rows", C, 1420.0, 300.0 / C, 50e-6, 0.0, step, n_dm, n_out)
    plan = dd.Plan.from_setup(s, dtype)
    d = oracle_table(s)
    x, _ = make_input(s, dtype, 22, plan.n_in + off)
    view = torch.from_numpy(x).cuda()[:, off:]
    ref, scale = oracle_window(d, x[:, off:], dtype, 0, n_dm, 0, n_out)
    for cfg in plan.configs():
        plan.select(cfg)
        got = plan.forward(view)
        assert plan.device_status() == 0, cfg
        assert_parity(got.cpu().numpy(), ref, scale, dtype, where=f"{dtype} offset {off} {cfg}")
