"""Marshalling of batched and served requests (mcubes._requests): the structures hold what one
mcubes_request built from each request's own arrays holds."""
import numpy as np
import pytest

from paper_2202_01753_gb300 import mcubes


def _values(a):
    """The fields of a request as Python values, the arrays read through its pointers."""
    return (a.integrand_id, a.params[:a.nparams], a.lo[:a.d], a.hi[:a.d], a.ncall, a.itmax, a.rel_tol, a.abs_tol, a.seed)


def test_scalars_are_one_element():
    reqs = [dict(fid=0, params=2.5, lo=-1.0, hi=np.float64(3.0), ncall=100, itmax=2),
            dict(fid=1, params=[1.0, 0.5, 0.25], lo=[0.0], hi=(1.0,), ncall=1e5, itmax=3, rel_tol=1e-3, abs_tol=2, seed=9),
            dict(fid=0, params=np.array(7), lo=0, hi=1, ncall=100, itmax=2)]
    arr, keep = mcubes._requests(reqs)
    assert [_values(a) for a in arr] == [(0, [2.5], [-1.0], [3.0], 100, 2, 0.0, 0.0, 0),
                                         (1, [1.0, 0.5, 0.25], [0.0], [1.0], 100000, 3, 1e-3, 2.0, 9),
                                         (0, [7.0], [0.0], [1.0], 100, 2, 0.0, 0.0, 0)]


def test_short_arrays_are_refused():
    """The library reads as many hi as lo values: the ones after a shorter hi are another request's."""
    ok = dict(fid=0, params=[1.0], lo=[0.0, 0.0], hi=[1.0, 1.0], ncall=100, itmax=2)
    for bad in (dict(hi=[1.0]), dict(hi=1.0), dict(hi=[]), dict(lo=np.zeros((2, 0))), dict(params=np.zeros((3, 0)))):
        for reqs in ([{**ok, **bad}], [{**ok, **bad}, ok], [ok, {**ok, **bad}]):
            with pytest.raises(ValueError):
                mcubes._requests(reqs)
    arr, _ = mcubes._requests([{**ok, "hi": [1.0, 2.0, 3.0]}])  # more than it reads
    assert _values(arr[0])[2:4] == ([0.0, 0.0], [1.0, 2.0])


def test_fid_is_an_integer():
    ok = dict(fid=0, params=[1.0], lo=[0.0], hi=[1.0], ncall=100, itmax=2)
    for fid in (1.0, 1.9, np.float64(2.0), "1", None):
        with pytest.raises(TypeError):
            mcubes._requests([{**ok, "fid": fid}])
    for fid in (1, np.int32(1), np.int64(1), True):
        assert mcubes._requests([{**ok, "fid": fid}])[0][0].integrand_id == 1
