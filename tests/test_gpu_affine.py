"""The FP64 affine families and table integrands, in the fixed-point form and just outside the rule
that selects it (csrc/affine.cu), against the oracle: boxes away from the unit
cube, few and many bins, sub-cube counts that are and are not powers of two,
ranges on both sides of the form's limits, negative and zero coefficients.
Tolerances: estimates within 1e-12 of the conditioning scale max(|I|, sum
|cube means| / m), variances within 1e-10 relative (differences of nearly equal
values), edges within 1e-12, as for the other double-precision runs."""
import numpy as np
import pytest

import oracle
from paper_2202_01753_gb300 import workloads as W

pytestmark = pytest.mark.gpu

G, C, O, P, A, D = W.F_GAUSS, W.F_CORNER, W.F_OSC, W.F_PRODPEAK, W.F_C0, W.F_DISCONT
CASES = [
    # family, params, lo, hi, ncall, nb, g
    ("gauss_d1", G, [2.0, 0.4, 0.2], [0.0], [1.0], 20_000, 500, 0),
    ("gauss_box", G, [0.5, 0.1, -2.0, 0.3, 0.9], [-1.0, -3.0], [1.5, 1.0], 20_000, 2, 0),
    ("gauss_d12", G, [1.0] + [0.5] * 12 + [0.2] * 12, [0.0] * 12, [1.0] * 12, 50_000, 300, 0),
    ("gauss_limit_in", G, [1.0, 0.5, 0.5 / (90.0 ** 0.5)], [0.0], [1.0], 30_000, 500, 0),
    ("gauss_limit_out", G, [1.0, 0.5, 0.5 / (9000.0 ** 0.5)], [0.0], [1.0], 30_000, 500, 0),
    ("gauss_negative", G, [-1.0, 0.5, 0.5, 0.2, 0.2], [0.0] * 2, [1.0] * 2, 20_000, 500, 0),
    ("corner_far", C, [0.5, 1.5, 2.0], [3.0, 0.0, 7.0], [3.5, 1.0, 9.0], 30_000, 1024, 7),
    ("corner_zero", C, [0.5, 0.0, 2.0], [0.0] * 3, [1.0] * 3, 30_000, 500, 0),
    ("osc_turns", O, [-3.75, 6.0, 0.01, 40.0], [-2.0, 0.0, 0.0], [2.0, 1.0, 1.0], 60_000, 64, 16),
    ("osc_negative", O, [0.2, -1.0, 2.0], [0.0] * 2, [1.0] * 2, 20_000, 500, 0),
    ("osc_many_turns", O, [0.2, 900.0], [0.0], [1.0], 20_000, 500, 0),
    ("prodpeak_box", P, [50.0, -8.0, 0.1, 0.4], [-0.2, 0.0], [0.6, 1.0], 30_000, 7, 5),
    ("prodpeak_sharp", P, [500.0, 0.5], [0.0], [1.0], 30_000, 500, 0),
    ("c0_box", A, [10.0, 3.0, 0.5, -0.25], [-1.0, -1.0], [1.0, 1.0], 30_000, 500, 3),
    ("c0_steep", A, [2000.0, 0.5], [0.0], [1.0], 30_000, 500, 0),
    ("discont", D, [5.0, 6.0, 0.4, 2.0], [0.0, 0.0], [1.0, 1.5], 30_000, 500, 0),
    ("discont_box", D, [5.0, 6.0, 0.4, 0.5], [-0.5, 0.0], [1.0, 1.0], 30_000, 500, 0),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("lanes", [0, 4])
def test_affine_against_oracle(gpu_ctx_factory, case, lanes):
    _, fid, params, lo, hi, ncall, nb, g = case
    params, lo, hi = np.array(params), np.array(lo), np.array(hi)
    o = oracle.integrate(fid, params, lo, hi, ncall, 4, ita=3, nb=nb, g_override=g, seed=21)
    ctx = gpu_ctx_factory(nbins=nb, ita=3, g_override=g, seed=21, lanes_per_cube=lanes)
    res = ctx.integrate(fid, params, lo, hi, ncall, 4)
    I, V = ctx.trace()
    grid = ctx.grid()
    ctx.close()
    pb = oracle.Problem(fid, params, lo, hi, ncall, nb=nb, g_override=g, seed=21)
    n = min(pb.m, 2000)
    sums, _, _, _ = pb.vsample(oracle.init_grid(pb.d, pb.nb), 0, False, 0, n)
    scale = max(np.max(np.abs(o["trace_I"])), sums[2] / n)
    assert res["iterations"] == 4
    np.testing.assert_allclose(I, o["trace_I"], rtol=0, atol=1e-12 * scale)
    np.testing.assert_allclose(V, o["trace_var"], rtol=1e-10, atol=0)
    np.testing.assert_allclose(grid, o["grid"], rtol=0, atol=1e-12)


_rng = np.random.default_rng(17)
TABLES = [dict(ndim=2, values=_rng.uniform(0.5, 2.0, (9, 33)), lo=(0.0, -1.0), hi=(1.0, 3.0)),
          dict(ndim=1, values=_rng.uniform(0.5, 2.0, 1000), lo=0.25, hi=0.75),
          dict(ndim=1, values=np.array([1.0, 3.0]), lo=-2.0, hi=5.0)]
TABLE_CASES = [
    # factors (table, axis, second axis), lo, hi: boxes inside, beside and across the knot ranges
    ("one_factor_each", [(0, 1, 0), (1, 2, -1), (2, 3, -1)], [-1.5, -0.5, 0.0, -3.0], [3.5, 1.5, 1.0, 6.0]),
    ("outside", [(1, 0, -1), (2, 1, -1)], [0.8, 7.0], [0.9, 8.0]),
    ("flat_axis", [(2, 1, -1)], [0.0, 0.0, 0.0], [1.0, 1.0, 1.0]),
    ("read_twice", [(0, 0, 1), (1, 0, -1)], [0.0, 0.0], [1.0, 1.0]),
    ("wide_box", [(1, 0, -1)], [-1e6, 0.0], [1e6, 1.0]),
    ("six_factors", [(2, j, -1) for j in range(6)], [0.0] * 6, [1.0] * 6),
]


@pytest.mark.parametrize("case", TABLE_CASES, ids=[c[0] for c in TABLE_CASES])
def test_tables_against_oracle(gpu_ctx_factory, case):
    _, factors, lo, hi = case
    params = np.array([-0.5, len(factors)] + [v for f in factors for v in f], dtype=np.float64)
    lo, hi = np.array(lo), np.array(hi)
    oracle.set_tables(TABLES)
    o = oracle.integrate(W.F_TABLE, params, lo, hi, 30_000, 4, nb=200, seed=22)
    ctx = gpu_ctx_factory(nbins=200, seed=22)
    ctx.set_tables(TABLES)
    ctx.integrate(W.F_TABLE, params, lo, hi, 30_000, 4)
    I, V = ctx.trace()
    ctx.close()
    np.testing.assert_allclose(I, o["trace_I"], rtol=0, atol=1e-12 * np.max(np.abs(o["trace_I"])))
    # a constant region's variance is rounding: beside the estimate's own last places
    np.testing.assert_allclose(V, o["trace_var"], rtol=1e-10, atol=1e-28 * np.max(o["trace_I"] ** 2))
