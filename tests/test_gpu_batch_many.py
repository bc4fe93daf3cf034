"""Batches with more integrals than the refinement launch has block rows (twice
the SM count): every block serves several integrals, its own finalisation of
one running ahead of other blocks' rebinning of the next.  Each integral's trace,
final grid and last histogram belong to the same, last iteration: against the
oracle within 1e-12 (edges; estimates relative), 1e-12 (variances) and 1e-11
of an axis's largest bin, as for the smaller batches (test_gpu_batch.py)."""
import numpy as np
import pytest

import oracle
from paper_2202_01753_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N, NB = 1000, 60


@pytest.mark.parametrize("rel_tol", [0.0, 0.05])
def test_last_iteration_is_whole(gpu_ctx_factory, rel_tol):
    """itmax or the tolerance ends the integrals: both are set by the finalising block."""
    rng = np.random.default_rng(31)
    reqs = []
    for i in range(N):
        d = int(rng.integers(2, 5))
        if i & 1:
            fid, params = W.F_CORNER, rng.uniform(0.5, 2.0, d)
        else:
            fid, params = W.F_GAUSS, np.concatenate([[1.0], rng.uniform(0.3, 0.7, d), rng.uniform(0.1, 0.3, d)])
        reqs.append(dict(fid=fid, params=params, lo=np.zeros(d), hi=np.ones(d), ncall=int(rng.integers(200, 900)),
                         itmax=3, rel_tol=rel_tol, abs_tol=0.0, seed=9000 + i))
    ctx = gpu_ctx_factory(nbins=NB)
    out = ctx.integrate_batch(reqs)
    its = set()
    for i, (r, b) in enumerate(zip(reqs, out)):
        o = oracle.integrate(r["fid"], r["params"], r["lo"], r["hi"], r["ncall"], 3, rel_tol=rel_tol, nb=NB,
                             seed=r["seed"])
        I, V, B, C = ctx.batch_trace(i, len(r["lo"]))
        its.add(b["iterations"])
        assert b["iterations"] == o["iterations"] == len(I), i
        np.testing.assert_allclose(I, o["trace_I"], rtol=1e-12, err_msg=str(i))
        np.testing.assert_allclose(V, o["trace_var"], rtol=1e-12, err_msg=str(i))
        np.testing.assert_allclose(B, o["grid"], rtol=0, atol=1e-12, err_msg=str(i))
        rowmax = np.abs(o["hist"]).max(axis=1, keepdims=True)
        assert np.max(np.abs(C - o["hist"]) / rowmax) <= 1e-11, i
    ctx.close()
    assert its == ({3} if rel_tol == 0.0 else {2, 3})
