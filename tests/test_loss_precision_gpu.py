"""The detection loss where boxcars nearly cancel their mean, against exact
rational arithmetic."""
import math
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _exact(row):
    """Mean, variance and boxcars of a row, as fractions."""
    v = [Fraction(float(x)) for x in row]
    b = [sum(v[t:t + 8]) for t in range(len(v) - 7)]
    mean = sum(b) / len(b)
    return mean, sum((x - mean) ** 2 for x in b) / len(b), b


def _run(x):
    from paper_1601_01165_gb300 import binding as dd
    t = torch.empty(x.shape, device="cuda")
    raw, g = dd.boxcar_snr(t.copy_(torch.from_numpy(x.copy())), grad=True)
    return dd.snr_result(raw), g.cpu().numpy()


# The squares about the mean are sums of two-float numbers (48 bits): the
# deviation has to come out to 2^-40, about 1e-12, however large the mean is.
@pytest.mark.parametrize("n", [10, 16, 100, 264, 1000])
@pytest.mark.parametrize("offset,noise", [(30.0, 1.0), (1e4, 1.0), (1e6, 0.1)])
def test_deviation_about_a_large_mean(n, offset, noise):
    rng = np.random.default_rng(n)
    row = (offset + noise * rng.standard_normal(n)).astype(np.float32)
    mean, var, b = _exact(row)
    r, _ = _run(row[None, :])
    sd = math.sqrt(var)
    assert r["valid"] == 1 and b[r["best_t"]] == max(b)
    assert abs(r["std"] / sd - 1.0) <= 2.0 ** -40
    # the mean is a double; the best boxcar's distance from it cancels down from |mean|
    assert abs(Fraction(r["mean"]) - mean) <= 32 * EPS * abs(mean)
    assert abs(r["snr"] - float((max(b) - mean)) / sd) <= 2.0 ** -40 * r["snr"] + 32 * EPS * abs(float(mean)) / sd
