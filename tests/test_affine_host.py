"""The double-precision affine families on the CPU: affine_prepare
(csrc/affine.cu) and the sampling code of both forms, built for the host
(tests/affine_host.cpp), against the same samples in long double."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2202_01753_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def affine(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("affine") / "affine_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-I", os.path.join(ROOT, "paper_2202_01753_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-I", cuda, "-o", exe, os.path.join(HERE, "affine_host.cpp")],
                   check=True)

    def run(op, fid, params, lo, hi, nb=500, g=2, n=1, power=1.0, axis=0, offset=0.0):
        vals = [op, fid, len(lo), nb, g, n, power, axis, offset] + [repr(float(v)) for v in (*params, *lo, *hi)]
        line = " ".join(str(v) for v in vals)
        return [float(v) for v in
                subprocess.run([exe], input=line + "\n", capture_output=True, text=True, check=True).stdout.split()]
    return run


@pytest.mark.parametrize("c0,others", [(1e-3, (6, 7)), (1e-6, (6, 7)), (1e-8, (60, 60)), (1e-10, (60, 60)),
                                       (2e-12, (60, 60)), (0.5, (6, 7)), (6.0, (5, 7)), (3.0, (200, 200))])
@pytest.mark.parametrize("power", [1.0, 3.0])
def test_discont_cut(affine, c0, others, power):
    """A cut 8 units of the last place of x to either side of a sample: in double precision x is good to
    1.5 such units (its cell's edge and the product rounded), so no sample changes sides."""
    _, wrong = affine("cut", W.F_DISCONT, [c0, *others, 0.5, 2.0, 2.0], [0.0] * 3, [1.0] * 3, g=5, n=4000, power=power,
                      offset=8.0)
    assert wrong == 0


def test_discont_ordinary_cuts_keep_the_fixed_form(affine):
    for w in (W.suite("f6", d) for d in (1, 6, 10)):
        assert affine("fix", w.fid, w.params, w.lo, w.hi)[0] == 1
    # cuts at or beyond the box's sides need no resolution
    for cut in (-0.5, 0.0, 1.0, 1.5):
        assert affine("fix", W.F_DISCONT, [1e-10, 60.0, cut, 0.5], [0.0] * 2, [1.0] * 2)[0] == 1


C0, CO, DI = W.F_C0, W.F_CORNER, W.F_DISCONT
MEANS = [(CO, [300.0] * 12), (CO, [600.0] * 6), (CO, [1300.0] * 3), (CO, [10.0] * 12), (CO, [11.0] * 11), (CO, [1.0] * 6),
         (CO, [126.0]), (C0, [40.0] * 12 + [0.0] * 12), (C0, [40.0] * 12 + [1.0] * 12), (C0, [40.0] * 11 + [0.0] * 11),
         (C0, [40.0] * 12 + [0.5] * 12), (C0, [170.0] * 3 + [0.0] * 3), (C0, [500.0, 0.0]),
         (DI, [40.0] * 12 + [2.0] * 12), (DI, [40.0] * 11 + [2.0] * 11), (DI, [170.0] * 3 + [0.9] * 3)]


@pytest.mark.parametrize("power", [1.0, 3.0])
@pytest.mark.parametrize("case", range(len(MEANS)))
def test_mean_error(affine, case, power):
    """The mean of F over 60,000 samples, even and corner-ward edges, at the ends of the form's ranges: relative
    error below one last place of a double, or the double-precision form's where that is larger."""
    fid, params = MEANS[case]
    d = len(params) if fid == CO else len(params) // 2
    _, err, err_double = affine("mean", fid, params, [0.0] * d, [1.0] * d, n=60000, power=power)
    assert abs(err) <= max(2.0 ** -52, abs(err_double))


def test_selection_at_the_limits(affine):
    """The cases that test_gpu_affine_limits.py runs take the fixed-point form, with the fraction bits that
    their rule ends at; just outside it is not taken."""
    from test_gpu_affine_limits import INSIDE
    bits = dict(gauss=52, osc=57, c0=54, corner=56, prodpeak=52, discont=54)
    for name, fid, params, d in INSIDE:
        assert affine("fix", fid, params, [0.0] * d, [1.0] * d) == [1, bits[name.split("_")[0]]], name
    for fid, params in ((W.F_GAUSS, [1.0, 0.0, 1.0 / (2.0 * 4100.0) ** 0.5]), (W.F_OSC, [0.3, 2.0 * np.pi * 65.0]),
                        (W.F_C0, [513.0, 0.0]), (W.F_CORNER, [128.0]), (W.F_PRODPEAK, [64.0, 0.0]),
                        (W.F_DISCONT, [513.0, 0.9])):
        assert affine("fix", fid, params, [0.0], [1.0])[0] == 0, (fid, params)
