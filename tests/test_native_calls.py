"""The native callers of the step's entry points against the same calls through ctypes (host functions, no GPU needed)."""
import os
import sysconfig

import numpy as np
import pytest


@pytest.fixture(params=["native", "ctypes"])
def binding(request, trj, monkeypatch):
    if request.param == "native":
        if not os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h")):
            pytest.skip("no Python headers: the binding stays with ctypes")
        assert trj._calls is not None, "binding/calls.cpp is not built"
    else:
        monkeypatch.setattr(trj, "_calls", None)
    monkeypatch.setattr(trj, "_step_calls", None)
    return request.param


def test_host_calls_give_the_same_tokens(trj, binding):
    context = np.array([5, 6, 7, 5, 6, 7, 5, 6], np.int32)
    draws = np.arange(10, dtype=np.int64) * 7919
    branches = trj.retrieve(context, 2, 3, draws)
    assert branches.shape == (2, 3) and branches[0].tolist() == [7, 5, 6]
    tokens, parent = np.array([6, 7, 5, 6], np.int32), np.array([-1, 0, 1, 2], np.int32)
    window = trj.refill_window(parent, tokens, 1, 3, context, draws[:3])
    assert window.shape == (3,) and window[:2].tolist() == [5, 6]


def test_errors_of_a_call_reach_the_caller(trj, binding):
    with pytest.raises(trj.TrjError):
        trj.retrieve(np.zeros(0, np.int32), 2, 3, np.zeros(6, np.int64))


def test_native_arguments_are_checked(trj, binding):
    if binding == "ctypes":
        pytest.skip("ctypes checks its own way")
    call = trj._fast().trj_retrieve
    for bad in [(1.5, 1, 1, 1, None, None), (b"", 1 << 31, 1, 1, None, None), (b"", 1, 1, 1, None, b"written to"), (b"", 1, 1, 1, None)]:
        with pytest.raises((TypeError, OverflowError)):
            call(*bad)


def test_a_module_that_is_built_but_does_not_load_is_an_error(trj, monkeypatch):
    if trj._calls is None:
        pytest.skip("not built")

    def broken(*_):
        raise ImportError("undefined symbol")
    monkeypatch.setattr(trj, "_lib", None)
    monkeypatch.setattr(trj.importlib, "import_module", broken)
    with pytest.raises(ImportError, match="undefined symbol"):
        trj.lib()
