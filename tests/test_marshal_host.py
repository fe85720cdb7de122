"""Host checks of the binding's argument marshalling that need no GPU: what its
Python path refuses."""
import types

import pytest
import torch

import paper_1902_08755_gb300 as ec
from paper_1902_08755_gb300 import api


def _shapes(h, w, pitch):
    """Depth buffers of the colour's pitch with too few rows, too few columns, or
    one dimension only, and one of another pitch."""
    buf = torch.ones((h, pitch))
    yield buf[:h - 1, :w]
    yield buf[:0, :w]
    yield buf[:, :w - 1]
    yield buf.reshape(-1)
    yield torch.ones((h, pitch + 1))[:, :w]


@pytest.mark.parametrize("pvp", [None, (2, 3, 9, 7)])
def test_output_depth_covers_the_output(monkeypatch, pvp):
    """Every row and column of the output rectangle is written, so the output
    depth has to have them."""
    monkeypatch.setattr(api, "_on_device", lambda *a: None)
    h, w, pitch = 7, 9, 12
    color = torch.zeros((h, pitch), dtype=torch.int32)[:, :w]
    good = torch.ones((h, pitch))[:, :w]
    assert api._target(color, good, pvp, 0).depth == good.data_ptr()
    assert api._target(color, torch.ones((h + 2, pitch)), pvp, 0).depth
    for bad in _shapes(h, w, pitch):
        with pytest.raises(ValueError):
            api._target(color, bad, pvp, 0)
    # a smaller rectangle needs only its own rows and columns
    small = torch.ones((h, pitch))[:4, :5]
    assert api._target(color, small, (0, 0, 5, 4), 0).depth == small.data_ptr()
    with pytest.raises(ValueError):
        api._target(color, small, (0, 0, 5, 5), 0)


class _Calls:
    """Stands in for the library: every entry point succeeds and is counted."""

    def __init__(self):
        self.names = []

    def __getattr__(self, name):
        return lambda *a: self.names.append(name) or 0


@pytest.fixture
def calls(monkeypatch):
    monkeypatch.setattr(api, "_on_device", lambda *a: None)
    lib = _Calls()
    monkeypatch.setattr(api, "_lib", lambda: lib)
    return lib.names


_CTX = types.SimpleNamespace(device=0, h=None)


@pytest.mark.parametrize("pvp", [None, (1, 2, 9, 7), (1, 2, 5, 4)])
def test_depth_gradients_cover_their_input(calls, pvp):
    """A gradient is written over its input's pvp."""
    h, w, pitch = 7, 9, 12
    color = torch.zeros((h, pitch, 4))[:, :w]
    im = ec.Image(color, pvp=pvp)
    ph, pw = (h, w) if pvp is None else (pvp[3], pvp[2])
    win, go = torch.zeros((h, w), dtype=torch.int16), torch.zeros((h, w, 4))

    def run(g):
        ec.composite_depth_backward(win, (0, 0, w, h), go, [im], [g], ctx=_CTX, stream=0)
    buf = torch.zeros((h, pitch, 4))
    run(buf[:, :w])
    run(buf[:ph, :pw])
    assert len(calls) == 2
    for bad in (buf[:ph - 1, :w], buf[:, :pw - 1]):
        with pytest.raises(ValueError):
            run(bad)
    assert len(calls) == 2
