"""Host checks of the binding's argument marshalling that need no GPU: what its
Python path refuses."""
import os
import subprocess
import sys
import types

import pytest
import torch

import paper_1902_08755_gb300 as ec
from paper_1902_08755_gb300 import api

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


_CHANGING_LISTS = r"""
import ctypes as C, gc, sys
import torch
from paper_1902_08755_gb300 import _abi as A

t = torch.zeros((4, 4), dtype=torch.int32)

class Clears:                                   # reading one of its attributes empties the lists
    def __init__(self, lists, attr):
        self.lists, self.attr, self.load = lists, attr, [bytearray(4096) for _ in range(8)]
    def __getattribute__(self, name):
        get = object.__getattribute__
        if name in ("color", "depth", "pvp", "roi"):
            if name == get(self, "attr"):
                for l in get(self, "lists"):
                    l.clear()
                gc.collect()
                junk = [bytearray(64) for _ in range(4096)]
            return t if name == "color" else None
        return get(self, name)

arr = (C.c_uint64 * 64)()
for attr in ("color", "pvp", "roi"):
    for _ in range(50):
        images = []
        images.append(Clears([images], attr))
        assert A.marshal().images(images, 0, 0, C.addressof(arr)) is False and not images
        images, grads = [], [torch.zeros((4, 4, 4))]
        images.append(Clears([images, grads], "color"))
        assert A.marshal().gradients(grads, images, 0, C.addressof(arr)) is False and not images and not grads
print("fine")
"""


def test_attributes_may_change_the_lists():
    """The images' attributes may be properties: code that takes the image (and
    its gradient) out of the lists while they are read."""
    r = subprocess.run([sys.executable, "-X", "dev", "-c", _CHANGING_LISTS], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "fine", (r.returncode, r.stdout, r.stderr[-2000:])
