"""Input rows of any stride: the shared-memory kernels copy spans on 16-byte
boundaries counted from the start of the input, so rows that start anywhere
between them (a tensor without row padding) must give the sums of padded rows,
down to the last samples of the last row, which no bulk copy may run past."""
import numpy as np
import pytest

from paper_1601_01165_gb300 import synth
from helpers import assert_parity, make_input, oracle_table, oracle_window

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "u8"])
@pytest.mark.parametrize("C,n_dm,n_out,step,pad", [
    (33, 9, 1001, 0.25, 0),       # n_in odd: every row starts at another offset
    (5, 1, 17, 0.0, 0),           # no delay: the last row is read to its last sample
    (40, 20, 2999, 0.0, 1),       # the same over several tiles and chunks
    (64, 70, 1503, 0.25, 2),
    (7, 16, 4096, 0.25, 3),
])
def test_any_row_stride_every_config(dtype, C, n_dm, n_out, step, pad):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("rows", C, 1420.0, 300.0 / C, 50e-6, 0.0, step, n_dm, n_out)
    plan = dd.Plan.from_setup(s, dtype)
    d = oracle_table(s)
    stride = plan.n_in + pad
    x, _ = make_input(s, dtype, 21, stride)
    # exactly the rows, with nothing of the tensor after the last sample
    xt = torch.from_numpy(x).cuda()
    assert xt.shape == (C, stride) and xt.stride(0) == stride
    ref, scale = oracle_window(d, x, dtype, 0, n_dm, 0, n_out)
    for cfg in plan.configs():
        plan.select(cfg)
        got = plan.forward(xt)
        torch.cuda.synchronize()
        assert plan.device_status() == 0, cfg
        assert_parity(got.cpu().numpy(), ref, scale, dtype, where=f"{dtype} stride {stride} {cfg}")
