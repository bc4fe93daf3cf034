"""The merge of single-precision partial histograms (fx_sum_floats,
csrc/fx_math.cuh), compiled for the host, against exact sums: nothing above
2^-100 of the largest addend is lost and the two words of the sum are rounded
to a double each, so the error stays below 2^-52 of the sum; non-finite addends
give what plain double additions give."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2202_01753_gb300", "csrc")


@pytest.fixture(scope="module")
def fxsum(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fx") / "fxsum_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "fxsum_host.cpp")],
                   check=True)

    def run(a, stride=1):
        a = np.asarray(a, np.float32)
        text = f"{stride} {len(a) // stride} " + " ".join(str(int(b)) for b in a.view(np.uint32))
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return float.fromhex(out.strip())
    return run


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 49, 456, 5000])
@pytest.mark.parametrize("span", [0, 10, 60, 252])
def test_sum_of_floats(fxsum, n, span):
    rng = np.random.default_rng(n * 1000 + span)
    a = np.ldexp(1.0 + rng.random(n), rng.integers(-span // 2, span // 2 + 1, n)).astype(np.float32)
    a[rng.random(n) < 0.1] = 0.0
    for v in (a, np.sort(a), np.sort(a)[::-1]):
        ref = math.fsum(v.astype(np.float64))
        assert abs(fxsum(v) - ref) <= ref * 2.0 ** -52


@pytest.mark.parametrize("a", [[0.0] * 9, [1e-45] * 20, [1e-45, 0.0, 3e-39], [3.4e38] * 30, [2.0 ** 100, 1e-45]])
def test_ends_of_the_range(fxsum, a):
    ref = math.fsum(np.asarray(a, np.float32).astype(np.float64))
    assert abs(fxsum(a) - ref) <= ref * 2.0 ** -52


def test_stride(fxsum):
    a = np.random.default_rng(1).random(11 * 5).astype(np.float32)
    ref = math.fsum(a[::5].astype(np.float64))
    assert abs(fxsum(a, 5) - ref) <= ref * 2.0 ** -52


def test_non_finite(fxsum):
    assert fxsum([1.0] * 12 + [np.inf]) == np.inf
    assert math.isnan(fxsum([np.nan] + [1.0] * 9))
