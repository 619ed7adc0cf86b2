"""The integer conversion of a float to a double (csrc/pair_convert.cuh) on the
CPU: every normal float exactly, infinities and NaN as themselves."""

import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def widen(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pair_convert") / "check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-o", exe,
                    os.path.join(ROOT, "tests", "pair_convert", "check_widen.cpp")], check=True)

    def run(x):
        bits = [f"{v:08x}" for v in np.asarray(x, dtype=np.float32).view(np.uint32)]
        out = subprocess.run([exe] + bits, check=True, capture_output=True, text=True).stdout.split()
        return np.array([int(v, 16) for v in out], dtype=np.uint64).view(np.float64)
    return run


def test_normal_floats_exactly(widen):
    f = np.finfo(np.float32)
    x = np.array([0.0, -0.0, 1.0, -1.5, 0.1, f.tiny, -f.tiny, f.max, -f.max, 2.0 ** 127], dtype=np.float32)
    assert np.array_equal(widen(x).view(np.uint64), x.astype(np.float64).view(np.uint64))
    x = np.random.Generator(np.random.PCG64(1)).integers(0x00800000, 0x7f800000, 500).astype(np.uint32).view(np.float32)
    assert np.array_equal(widen(x), x.astype(np.float64))


def test_subnormals_give_zero(widen):
    assert np.array_equal(widen([1e-40, -1e-45]), [0.0, 0.0])


def test_infinities_and_nan_stay(widen):
    w = widen([np.inf, -np.inf, np.nan, -np.nan])
    assert w[0] == np.inf and w[1] == -np.inf and np.all(np.isnan(w[2:]))
