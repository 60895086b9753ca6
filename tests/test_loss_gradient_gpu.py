"""The detection loss's gradient where its terms cancel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(x):
    from paper_1601_01165_gb300 import binding as dd
    t = torch.empty(x.shape, device="cuda")
    raw, g = dd.boxcar_snr(t.copy_(torch.from_numpy(x.copy())), grad=True)
    return dd.snr_result(raw), g.cpu().numpy()


# Two starts have S/N 1 whatever the samples, so their gradient is zero, and
# exactly so where mean and deviation are exact.
def test_gradient_of_two_exact_starts_is_zero():
    rng = np.random.default_rng(3)
    for _ in range(100):
        row = rng.integers(20, 2000, 9).astype(np.float32)
        if row[0] == row[8]:
            continue
        r, g = _run(row[None, :])
        assert r["valid"] == 1 and r["snr"] == 1.0 and (g == 0).all(), row
