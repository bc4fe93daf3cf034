"""The largest bin counts of the double-precision batched path: 12 axes of 803
bins (cells and histogram of one block, 231,264 bytes) run, as in the
single-integral path, whatever the dimensions of the requests."""
import numpy as np
import pytest

import oracle
from paper_2202_01753_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [801, 803])
def test_largest_grids(gpu_ctx_factory, nb):
    reqs = [dict(fid=W.F_CORNER, params=np.linspace(0.5, 2.0, d), lo=np.zeros(d), hi=np.ones(d), ncall=9000, itmax=3,
                 seed=60 + d) for d in (2, 11, 12)]
    ctx = gpu_ctx_factory(nbins=nb)
    out = ctx.integrate_batch(reqs)
    for i, r in enumerate(reqs):
        d = len(r["lo"])
        o = oracle.integrate(r["fid"], r["params"], r["lo"], r["hi"], r["ncall"], 3, nb=nb, seed=r["seed"])
        I, V, B, _ = ctx.batch_trace(i, d)
        np.testing.assert_allclose(I, o["trace_I"], rtol=1e-12)
        np.testing.assert_allclose(V, o["trace_var"], rtol=1e-12)
        np.testing.assert_allclose(B, o["grid"], rtol=0, atol=1e-12)
    ctx.close()
    assert len(out) == 3
