"""The float pair that the mixed mode stores a state's q-variables as when it is set
(csrc/pair_convert.cuh, nearest_pair), on the CPU."""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_pair_is_within_half_a_unit_of_its_low_word(tmp_path):
    """|lo| is at most 2^-24 of x and its rounding 2^-25 of that: 2^-49. (A truncated
    leading word leaves 2^-48.)"""
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-o", exe,
                    os.path.join(ROOT, "tests", "pair_convert", "check_nearest.cpp")], check=True)
    worst = float(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    assert 0.5 < worst <= 1.0
