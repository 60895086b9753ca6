"""The few-row weight gradient with samples that are not finite in many
channels at once: every block of the kernel that looks for them finds one, in
several waves of blocks, and all later kernels have to agree on what it found."""
import numpy as np
import pytest

from paper_1601_01165_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1, 3])
def test_non_finite_samples_in_many_channels(step):
    from paper_1601_01165_gb300 import binding as dd
    s = synth.Setup("bad", 4096, 1420.0, 300.0 / 4096, 50e-6, 0.0, 0.01, 20, 5000)
    plan = dd.Plan.from_setup(s, "f32")
    assert "tmw9_f32_d9_t4096" in plan.configs()
    x = plan.alloc_input()
    x[:, :plan.n_in] = 1.0
    # at different places, so that blocks find them at different times
    at = torch.arange(0, s.channels, step, device="cuda")
    x[at, (at * 37) % (s.n_out - 100) + plan.max_delay] = float("inf")
    g = torch.zeros((s.n_dm, s.n_out), device="cuda")
    g[7, ::2] = 1.0
    want = np.where(np.arange(s.channels) % step == 0, np.nan, np.float32(s.n_out // 2)).astype(np.float32)
    for _ in range(5):
        _, gw = plan.adjoint(g, x=x, grad_in=False, grad_w=True)
        assert plan.device_status() == 0
        np.testing.assert_array_equal(gw.cpu().numpy(), want)
