"""Which kernels compute the weight gradient alone, told by what they round: a
row of 2^24, 1, -2^24 four samples apart is within one float chain of the tiles
(every fourth of 32 samples), which lose the 1, and in three threads of the
few-row kernel, which adds them in double."""
import pytest

from paper_1601_01165_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_dm,n_rows,few", [(40, 1, True), (40, 8, True), (40, 9, False), (15, 8, False), (16, 8, True),
                                             (2, 1, True), (1, 1, False)])
def test_few_rows_go_to_their_own_kernel(n_dm, n_rows, few):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("route", 130, 1420.0, 2.0, 50e-6, 0.0, 0.25, n_dm, 3001)
    plan = dd.Plan.from_setup(s, "f32")
    assert "tmw9_f32_d9_t4096" in plan.configs()
    x = plan.alloc_input()
    x[:, :plan.n_in] = 1.0
    g = torch.zeros((n_dm, s.n_out), device="cuda")
    g[n_dm - n_rows:, 2000] = 1.0
    g[n_dm - 1, 64], g[n_dm - 1, 68], g[n_dm - 1, 72] = 2.0 ** 24, 1.0, -2.0 ** 24
    _, gw = plan.adjoint(g, x=x, grad_in=False, grad_w=True)
    assert plan.device_status() == 0
    exact = float(n_rows + 1)
    assert ((gw == exact) if few else (gw == exact - 1.0)).all(), gw
