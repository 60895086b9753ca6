"""The detection loss of the shortest rows: one and two boxcar starts."""
import math
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


# One start has no deviation, whatever its eight samples: no S/N, no gradient.
def test_rows_of_one_start_have_no_snr():
    rng = np.random.default_rng(1)
    x = rng.standard_normal((200, 8)) * 2.0 ** (rng.random((200, 8)) * 30)
    for row in x.astype(np.float32):
        r, g = _run(row[None, :])
        assert r["valid"] == 0 and (g == 0).all(), row


# Two starts that differ are one deviation above and below their mean, to what
# the double mean of two boxcars can tell (2^-50 of the samples, in deviations)
# and the square of what two-float boxcars can (2^-47).
def test_rows_of_two_starts_have_snr_one():
    rng = np.random.default_rng(2)
    x = (rng.standard_normal((200, 9)) * 2.0 ** (rng.random((200, 9)) * 30)).astype(np.float32)
    for row in x:
        _, var, b = _exact(row)
        rel = float(np.abs(row).astype(np.float64).sum()) / math.sqrt(var)
        if b[0] == b[1] or 2.0 ** -47 * rel > 1e-3:
            continue
        r, _ = _run(row[None, :])
        assert r["valid"] == 1
        assert abs(r["snr"] - 1.0) <= 2.0 ** -50 * rel + (2.0 ** -47 * rel) ** 2 + 1e-14, row
