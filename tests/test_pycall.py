"""The C module behind the per-token calls (csrc/pycall.c): argument checks and conversions, without a GPU.  Every call here
hands the library a null handle or null vectors, which it refuses before it touches anything."""
import ctypes

import pytest

from paper_2607_21985_b200 import build, spdp


@pytest.fixture(scope="module")
def L():
    build.build()
    return spdp.lib()


def test_status_comes_back(L):
    assert L.call_spmspv(None, 1 << 47, 1, 0.5, None, 1 << 47, 0, 0) == spdp.SPDP_ERR_INVALID_ARG
    assert L.call_spmspv_batch(None, 16, 1, 1, 0, 0.0, None, 0, 16, 1, 0, None) == spdp.SPDP_ERR_INVALID_ARG
    assert L.call_spmm(None, 16, 1, 1, 16, 1, 0, 0) == spdp.SPDP_ERR_INVALID_ARG
    assert L.call_swiglu_dp(None, None, 5, 0.5, None, None, None, None) == spdp.SPDP_ERR_INVALID_ARG


@pytest.mark.parametrize("name,n", [("spmspv", 8), ("spmspv_batch", 12), ("spmm", 8), ("swiglu_dp", 8)])
def test_wrong_arguments_raise(L, name, n):
    call = getattr(L, "call_" + name)
    with pytest.raises(TypeError):
        call(*[0] * (n - 1))
    with pytest.raises(TypeError):
        call(*[0] * (n + 1))
    with pytest.raises(TypeError):
        call("x", *[0] * (n - 1))
    with pytest.raises((TypeError, OverflowError)):
        call(1 << 70, *[0] * (n - 1))


def test_arguments_arrive(L):
    """A callback in place of the entry point sees what was passed."""
    from paper_2607_21985_b200 import _pycall
    seen = []
    sig = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_float, ctypes.c_void_p, ctypes.c_void_p,
                           ctypes.c_int, ctypes.c_void_p)
    cb = sig(lambda *a: seen.append(a) or -3)
    assert _pycall.spmspv(ctypes.cast(cb, ctypes.c_void_p).value, 5, (1 << 64) - 16, 2, -0.25, None, 7, 1, 0) == -3
    assert seen == [(5, (1 << 64) - 16, 2, -0.25, None, 7, 1, None)]
    with pytest.raises(OverflowError):
        _pycall.spmspv(ctypes.cast(cb, ctypes.c_void_p).value, 5, 6, 1 << 40, 0.0, None, 7, 1, 0)


def test_ctypes_values_are_taken_as_ctypes_takes_them(L):
    """A handle or stream kept as a ctypes value (or an object that names its own) goes through as it does through ctypes itself."""
    from paper_2607_21985_b200 import _pycall
    seen = []
    vp, ci = ctypes.c_void_p, ctypes.c_int
    sig = ctypes.CFUNCTYPE(ci, vp, vp, ci, ctypes.c_float, vp, vp, ci, vp)
    cb = sig(lambda *a: seen.append(a) or 0)

    class Stream:
        _as_parameter_ = 99
    args = (vp(5), 6, ci(2), 0.5, vp(None), vp(7), 1, Stream())
    assert cb(*args) == 0 and _pycall.spmspv(ctypes.cast(cb, vp).value, *args) == 0
    assert seen == [(5, 6, 2, 0.5, None, 7, 1, 99)] * 2
    for bad in ("x", b"x", 5.0, vp, object(), ctypes.c_float(1.0)):
        with pytest.raises(TypeError):
            _pycall.spmspv(ctypes.cast(cb, vp).value, bad, *args[1:])
    assert len(seen) == 2


def test_module_belongs_to_this_interpreter(L):
    """A module built for another Python is neither imported nor taken for up to date."""
    import importlib.machinery
    import os
    from paper_2607_21985_b200 import _pycall
    suffix = importlib.machinery.EXTENSION_SUFFIXES[0]
    assert "cpython" in suffix and os.path.basename(build.PYCALL) == "_pycall" + suffix
    assert os.path.samefile(_pycall.__file__, build.PYCALL)
