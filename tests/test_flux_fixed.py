"""The fixed-point form of the split-flux differences with large steps
(csrc/flux_fixed.cuh) on the CPU, against binary128 and a plain double
evaluation, and its tables against their generator."""

import importlib.util
import os
import platform
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_07031_gb300", "csrc")


@pytest.fixture(scope="module")
def measured(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("flux_fixed") / "check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "flux_pair", "check_flux_fixed.cpp")]
                   + (["-lquadmath"] if platform.machine() == "x86_64" else []), check=True)

    def run(mach, log2_step, pairs=2000):
        out = subprocess.run([exe, str(mach), str(log2_step), str(pairs)], check=True,
                             capture_output=True, text=True).stdout.split()
        return int(out[0]), [float(v) for v in out[1:5]], [float(v) for v in out[5:9]]
    return run


@pytest.mark.parametrize("mach", [0.0, 0.3, 0.85, 2.0, 4.5])
@pytest.mark.parametrize("log2_step", [-30, -6, -3, 0])
def test_difference_error(measured, mach, log2_step):
    """Factors, moments, the first product and the difference are each rounded
    once, by half of 2^-52 at most: 2^-52 of G in the 2-norm. A plain double
    evaluation with a moving gas is no nearer."""
    taken, err, err64 = measured(mach, log2_step)
    assert taken == 2000 or (mach == 4.5 and taken > 1500)
    assert max(err) < 2.0 ** -52
    assert mach == 0.0 or all(a <= b for a, b in zip(err, err64))


def test_states_out_of_range_are_left_out(measured):
    """|S| beyond the table of erfcx (most states at Mach 40): refused."""
    assert measured(40.0, 0)[0] < 60


def test_tables_match_their_generator(tmp_path):
    pytest.importorskip("mpmath")
    spec = importlib.util.spec_from_file_location("gen_fixed_tables",
                                                  os.path.join(CSRC, "gen_fixed_tables.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    out = tmp_path / "fixed_tables.h"
    gen.main(str(out))
    with open(os.path.join(CSRC, "fixed_tables.h")) as f:
        assert out.read_text() == f.read()
