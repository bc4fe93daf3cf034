"""The fixed-point functions of the FP64 kernels' affine families
(csrc/fx_math.cuh), compiled for the host (tests/fxfixed_host.cpp), against
40-digit references at the ends of their table intervals, at their largest and
smallest arguments and in between.  Tolerances follow from the construction:
the exponential's reduced argument is exact to 2^-61 and its result rounded
once (2^-53, doubled for the tables); the reciprocal is good to 2^-60; the
cosine to 2^-60 absolute."""
import os
import shutil
import subprocess

import mpmath
import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2202_01753_gb300", "csrc")


@pytest.fixture(scope="module")
def fxfixed(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fx") / "fxfixed_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "fxfixed_host.cpp")],
                   check=True)

    def run(op, us, f=0):
        lines = "".join(f"{op} {u} {f}\n" for u in us)
        return subprocess.run([exe], input=lines, capture_output=True, text=True, check=True).stdout.split()
    return run


def _u64s(rng, n, bits=64):
    return [int(x) >> (64 - bits) for x in rng.integers(0, 2 ** 64, n, dtype=np.uint64)]


@pytest.mark.parametrize("neg", [True, False])
@pytest.mark.parametrize("fq", [52, 55, 58, 62])
def test_exp_fixed(fxfixed, neg, fq):
    mpmath.mp.dps = 40
    top = min(2 ** 64, 708 << fq) - 1
    us = [int(u * top) for u in np.random.default_rng(5).random(3000)] + [0, 1, top]
    ln = mpmath.log(2) / 256
    for k in range(1, 700, 7):  # next to the multiples of ln2/256, where n changes
        b = int(mpmath.nint(k * ln * 2 ** fq))
        us += [b - 1, b, b + 1]
    us = [u for u in us if 0 <= u <= top]
    got = fxfixed("e" if neg else "E", us, fq)
    for u, v in zip(us, got):
        y = mpmath.mpf(u) / 2 ** fq
        ref = mpmath.exp(-y if neg else y)
        assert abs(mpmath.mpf(float.fromhex(v)) - ref) <= ref * mpmath.mpf(2) ** -52, (u, v)


def test_exp_fixed_underflow(fxfixed):
    assert set(fxfixed("e", [746 << 52, 2 ** 64 - 1], 52)) == {"0x0p+0"}


def test_recip(fxfixed):
    rng = np.random.default_rng(6)
    us = [2 ** 63 | u for u in _u64s(rng, 4000, 63)]
    us += [2 ** 63, 2 ** 63 + 1, 2 ** 64 - 1, 2 ** 64 - 2 ** 40, 2 ** 64 - 2 ** 41]
    us += [2 ** 63 + (k << 55) + e for k in range(256) for e in (0, 1, (1 << 40) - 1)]
    for u, v in zip(us, fxfixed("r", us)):
        assert abs(int(v) * u - 2 ** 127) <= 2 ** 127 >> 60, (u, v)
        assert 2 ** 63 <= int(v) < 2 ** 64


def test_cos_turns(fxfixed):
    mpmath.mp.dps = 40
    rng = np.random.default_rng(7)
    us = _u64s(rng, 4000)
    us += [(k << 54) + e for k in range(0, 1024, 5) for e in (0, 1, (1 << 54) - 1)]
    us += [0, 1, 2 ** 62, 2 ** 62 - 1, 2 ** 62 + 1, 2 ** 63, 2 ** 63 - 1, 3 * 2 ** 62, 3 * 2 ** 62 + 1, 2 ** 64 - 1]
    for u, v in zip(us, fxfixed("c", us)):
        ref = mpmath.cos(2 * mpmath.pi * mpmath.mpf(u) / 2 ** 64)
        assert abs(mpmath.mpf(int(v)) / 2 ** 63 - ref) <= mpmath.mpf(2) ** -60, (u, v)
