"""The adjoint in the checked build (see test_checked_gpu.py): float grouped sums,
which only the transposed plan has, and every route of the weight gradient."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_checked_build_runs_adjoints_in_range():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_01165_gb300 import build
    env = dict(os.environ, DD_LIBRARY=build.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked_adjoint_run.py")], env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "in range and equal to the oracle" in r.stdout
