"""Training calls refuse a missing or bad input norm, and every other bad argument, with a status
before they touch a device (no GPU needed)."""
import ctypes as ct
import math

import pytest

import paper_cs_0703028_gb300 as rt

D = ct.c_void_p(16)  # a device address that is never read: the checks come first


def _norm(lo=0.0, hi=1.0, scale=1.0):
    return rt.rt_mlp_norm((ct.c_float * 4)(*[lo] * 4), (ct.c_float * 4)(*[hi] * 4), 0.0, scale)


def _steps(norm, batch=64, n_steps=2, params=D, adam=D):
    return rt.lib().rt_mlp_train_steps(params, adam, adam, D, D, D, 256, batch, norm, 1e-3, 1e-4, 1, n_steps, 100, None, None, None)


# batches of one tile, of several, and more rows than there are
@pytest.mark.parametrize("batch", [1, 128, 200])
def test_bad_norms_are_refused(batch):
    assert _steps(None, batch) == rt.RT_E_INVAL
    assert b"norm" in rt.lib().rt_last_error()
    for bad in (_norm(hi=0.0), _norm(lo=math.nan), _norm(hi=math.inf), _norm(scale=0.0), _norm(scale=math.nan)):
        assert _steps(ct.byref(bad), batch) == rt.RT_E_INVAL
    L = rt.lib()
    assert L.rt_mlp_train_steps_nets(4, D, D, D, D, D, D, 256, batch, None, 1e-3, 1e-4, 1, 2, 100, None, None, None) == rt.RT_E_INVAL
    assert L.rt_mlp_train_step(D, D, D, D, D, D, batch, None, 1e-3, 1, 0, D, None, None) == rt.RT_E_INVAL


def test_bad_buffers_are_refused():
    good = _norm()
    assert _steps(ct.byref(good), params=None) == rt.RT_E_INVAL
    assert _steps(ct.byref(good), adam=None) == rt.RT_E_INVAL
    assert _steps(ct.byref(good), batch=300) == rt.RT_E_INVAL
    assert _steps(None, n_steps=0) == 0  # nothing to do: nothing is read
