"""The range of sizes that the float-pair form (csrc/flux_pair.cuh) accepts, on the
CPU against binary128: beta and ln(rho beta^2.5) reach their ends together."""

import os
import platform
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_accepted_state_is_held(tmp_path):
    """At the corners the moments E beta^-3 .. E beta^-4 leave the floats' range:
    such states are refused, and what is taken has finite differences, each
    within 2^-46 of G at a step of 2^-10 (the form's 2^-43 of dG, with 2^-8 for
    |S| = 4, where G moves by up to 16 times the step)."""
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "flux_pair", "check_pair_range.cpp")]
                   + (["-lquadmath"] if platform.machine() == "x86_64" else []), check=True)
    taken, bad, worst = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert int(bad) == 0
    assert int(taken) > 5000
    assert float(worst) < 2.0 ** -46
