"""The mixed mode's FP32 split-flux differences (csrc/flux_mixed.cuh) on the CPU
against binary128: the form in S, which gamma = 1.4 takes, is no further off than
the primitive differences that it stands in for."""

import os
import platform
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def measured(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("flux_mixed") / "check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "flux_pair", "check_flux_mixed.cpp")]
                   + (["-lquadmath"] if platform.machine() == "x86_64" else []), check=True)

    def run(mach, log2_step, pairs=4000):
        out = subprocess.run([exe, str(mach), str(log2_step), str(pairs)], check=True,
                             capture_output=True, text=True).stdout.split()
        return int(out[0]), [float(v) for v in out[1:5]], [float(v) for v in out[5:9]]
    return run


@pytest.mark.parametrize("mach", [0.0, 0.3, 0.63, 0.85])
@pytest.mark.parametrize("log2_step", [-3, -6, -10, -14])
def test_difference_error(measured, mach, log2_step):
    taken, err, prim = measured(mach, log2_step)
    assert taken > 3900
    assert all(a <= b for a, b in zip(err, prim)), (err, prim)
