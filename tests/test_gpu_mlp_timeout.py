"""Training after a pass that gave up one of its bounded waits: the parameters, the
moments and the step count stay those of the last good step."""

import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2108_07031_gb300 import build as B  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_timed_out_step_changes_nothing(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.run([B._nvcc()] + B.ARCH + ["-O2", "-std=c++17", "-o", exe,
                   os.path.join(ROOT, "tests", "mlp_timeout", "check_timeout.cu")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout + out.stderr
