"""The FP64 affine families at the ends of the fixed-point form's ranges (csrc/affine.cu), against the
oracle: estimates within 1e-12 of the conditioning scale max(|I|, sum |cube
means| / m), variances within 1e-10 relative and edges within 1e-12, as in
test_gpu_affine.py."""
import numpy as np
import pytest

import oracle
from paper_2202_01753_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def against_oracle(make_ctx, fid, params, lo, hi, ncall, nb=500):
    params, lo, hi = np.array(params, dtype=float), np.array(lo, dtype=float), np.array(hi, dtype=float)
    o = oracle.integrate(fid, params, lo, hi, ncall, 3, nb=nb, seed=23)
    ctx = make_ctx(nbins=nb, seed=23)
    ctx.integrate(fid, params, lo, hi, ncall, 3)
    I, V = ctx.trace()
    grid = ctx.grid()
    ctx.close()
    pb = oracle.Problem(fid, params, lo, hi, ncall, nb=nb, seed=23)
    n = min(pb.m, 2000)
    sums, _, _, _ = pb.vsample(oracle.init_grid(pb.d, pb.nb), 0, False, 0, n)
    scale = max(np.max(np.abs(o["trace_I"])), sums[2] / n)
    np.testing.assert_allclose(I, o["trace_I"], rtol=0, atol=1e-12 * scale)
    np.testing.assert_allclose(V, o["trace_var"], rtol=1e-10, atol=0)
    np.testing.assert_allclose(grid, o["grid"], rtol=0, atol=1e-12)


@pytest.mark.parametrize("c0", [1e-3, 1e-6, 1e-8, 1e-10, 2e-12])
@pytest.mark.parametrize("c1", [6.0, 60.0])
def test_discont_flat_axis(gpu_ctx_factory, c0, c1):
    """A cut on an axis whose coefficient is small beside the others' (off the bin edges)."""
    against_oracle(gpu_ctx_factory, W.F_DISCONT, [c0, c1, 0.4001234567, 2.0], [0.0] * 2, [1.0] * 2, 1_000_000)


# just inside each rule (csrc/affine.cu): the least fraction bits and the largest sums that an integral
# whose F^2 neither overflows nor leaves an axis to subnormal sums can have
INSIDE = [
    ("gauss_4000_d1", W.F_GAUSS, [1.0, 0.0, 1.0 / (2.0 * 4000.0) ** 0.5], 1),
    ("osc_60_turns", W.F_OSC, [0.3, 2.0 * np.pi * 60.0], 1),
    ("osc_60_turns_d3", W.F_OSC, [0.3] + [2.0 * np.pi * 60.0] * 3, 3),
    ("c0_300_d1", W.F_C0, [300.0, 0.0], 1),
    ("c0_300_d12", W.F_C0, [25.0] * 12 + [0.0] * 12, 12),
    ("corner_127", W.F_CORNER, [126.0], 1),
    ("corner_121_d12", W.F_CORNER, [10.0] * 12, 12),
    ("prodpeak_4000", W.F_PRODPEAK, [63.2, 0.0], 1),
    ("prodpeak_4000_d3", W.F_PRODPEAK, [63.2] * 3 + [0.0] * 3, 3),
    ("discont_300_d1", W.F_DISCONT, [300.0, 0.9], 1),
    ("discont_300_d12", W.F_DISCONT, [25.0] * 12 + [0.9] * 12, 12),
]


@pytest.mark.parametrize("case", INSIDE, ids=[c[0] for c in INSIDE])
def test_inside_the_limits(gpu_ctx_factory, case):
    _, fid, params, d = case
    against_oracle(gpu_ctx_factory, fid, params, [0.0] * d, [1.0] * d, 60_000)
