"""The float-pair layout of a cloud (csrc/lskum_setup.cpp) on the CPU: hi + lo + rest
is the double, and clouds of sizes that floats do not hold are told apart."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pair_layout") / "check")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=gnu++17", "-o", exe,
                    os.path.join(ROOT, "tests", "pair_convert", "check_split.cpp")], check=True)
    return lambda *a: int(subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout)


def test_pairs_with_their_rests_are_the_doubles(check):
    """A million doubles of either sign, 2^-60 to 2^60."""
    assert check() == 0


@pytest.mark.parametrize("log2_scale, held", [(-140, 0), (-60, 0), (-31, 0), (-20, 1), (0, 1), (20, 1), (31, 0), (60, 0),
                                              (140, 0)])
def test_sizes_that_the_pair_form_takes(check, log2_scale, held):
    assert check(log2_scale) == held
