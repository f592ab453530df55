"""The torch conveniences look torch and the library's function up once (no GPU needed: CUDA initialisation is replaced)."""
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
