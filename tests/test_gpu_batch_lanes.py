"""lanes_per_cube on batches whose cubes hold fewer samples than lanes, or a
number that is no power of two: every sample is drawn once, so that traces
agree with the oracle within 1e-12 and the last histogram within 1e-11 of an
axis's largest bin, as for the other double-precision batches."""
import numpy as np
import pytest

import oracle
from paper_2202_01753_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 2, 4, 8, 32])
def test_batch_lanes_against_oracle(gpu_ctx_factory, lanes):
    rng = np.random.default_rng(32)
    reqs = []
    for p in (2, 3, 5, 7, 9, 33):  # samples per cube
        for d, g in ((1, 70), (3, 6), (5, 4)):
            reqs.append(dict(fid=W.F_CORNER, params=rng.uniform(0.5, 2.0, d), lo=np.zeros(d), hi=np.ones(d),
                             ncall=p * g ** d, itmax=3, seed=50 + p))
    for g in (70, 6, 4):
        d = {70: 1, 6: 3, 4: 5}[g]
        mine = [r for r in reqs if len(r["lo"]) == d]
        ctx = gpu_ctx_factory(nbins=100, g_override=g, lanes_per_cube=lanes)
        out = ctx.integrate_batch(mine)
        for i, (r, b) in enumerate(zip(mine, out)):
            o = oracle.integrate(r["fid"], r["params"], r["lo"], r["hi"], r["ncall"], 3, nb=100, g_override=g,
                                 seed=r["seed"])
            assert (b["g"], b["p"]) == (o["g"], o["p"]) == (g, r["ncall"] // g ** d)
            I, V, _, C = ctx.batch_trace(i, d)
            np.testing.assert_allclose(I, o["trace_I"], rtol=1e-12)
            np.testing.assert_allclose(V, o["trace_var"], rtol=1e-12)
            assert np.max(np.abs(C - o["hist"]) / o["hist"].max(axis=1, keepdims=True)) <= 1e-11
        ctx.close()
