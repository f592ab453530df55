"""The torch conveniences look torch and the library's function up once (no GPU needed: CUDA initialisation is replaced)."""
import ctypes
import os
import sys

import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from paper_2605_29843_b200 import build as harp_build


@pytest.fixture
def unbound(monkeypatch):
    harp_build.build()
    for name in ("_apply_ex", "_raw_stream", "_current_device"):
        monkeypatch.setattr(harp, name, None)


def test_nothing_is_published_before_cuda_is_up(unbound, monkeypatch):
    """Another thread that calls in the meantime must find everything bound, or nothing."""
    seen = []
    monkeypatch.setattr(torch.cuda, "init", lambda: seen.append(harp._apply_ex))
    harp._bind_torch()
    assert seen == [None]
    assert harp._apply_ex is not None and harp._raw_stream is not None and harp._current_device is not None


def test_a_failed_initialisation_is_tried_again(unbound, monkeypatch):
    def fail():
        raise RuntimeError("no driver")
    monkeypatch.setattr(torch.cuda, "init", fail)
    with pytest.raises(RuntimeError):
        harp._bind_torch()
    assert harp._apply_ex is None
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    harp._bind_torch()
    assert harp._apply_ex is not None


def test_the_call_without_ctypes_takes_what_ctypes_took(unbound, monkeypatch):
    """None for a null pointer, anything with __index__ for an integer; floats and a wrong number of arguments are refused."""
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    harp._bind_torch()
    null, bad_dtype = 1, harp.lib().harp_apply_ex(1, 1, 1, 7, 0, 0, None)
    assert harp._apply_ex(None, 1 << 63, np.int64(1), 0, 0, np.int32(0), None) == null
    assert harp._apply_ex(1, 1, 1, 7, 0, 0, 0) == bad_dtype != null
    for args in ((None, 0, 1.0, 0, 0, 0, 0), (None, 0, 1, 0, 0, 0), (None, 0, 1, 0, 0, "0", 0)):
        with pytest.raises(TypeError):
            harp._apply_ex(*args)


def test_a_tree_with_the_library_alone_calls_through_ctypes(unbound, monkeypatch):
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setitem(sys.modules, harp.__name__ + "._harpcall", None)       # as if it were not there
    monkeypatch.delattr(harp, "_harpcall", raising=False)
    harp._bind_torch()
    assert harp._apply_ex is harp.lib().harp_apply_ex
    assert harp._apply_ex(None, 0, 1, 0, 0, 0, None) == 1


def test_the_call_is_built_for_every_interpreter():
    """The stable interface, and a name that no other interpreter's build has."""
    harp_build.build()
    assert os.path.basename(harp_build.CALL) == "_harpcall.abi3.so" and os.path.exists(harp_build.CALL)
    assert harp._without_ctypes(harp.lib().harp_apply_ex)(None, 0, 1, 0, 0, 0, None) == 1
    assert "Py_LIMITED_API" in open(harp_build.CALL_SRC).read()


@pytest.mark.parametrize("at", [2, 3, 4, 5])
def test_none_is_no_number(unbound, monkeypatch, at):
    """Rows, codes and the direction, as ctypes refuses them; the plan, the rows' address and the stream are pointers."""
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    harp._bind_torch()
    args = [None, None, 1, 0, 0, 0, None]
    args[at] = None
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        harp._apply_ex(*args)
