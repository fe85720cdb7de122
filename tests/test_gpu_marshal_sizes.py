"""The native marshalling takes no buffer that is smaller than what a call
writes or reads: such calls are refused before anything is launched."""
import ctypes as C

import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu
from paper_1902_08755_gb300 import _abi as A
from paper_1902_08755_gb300 import api

pytestmark = pytest.mark.gpu


def test_output_depth_covers_the_output():
    require_gpu()
    h, w, pitch = 7, 9, 12
    color = torch.zeros((h, pitch), dtype=torch.int32, device="cuda")[:, :w]
    buf = torch.ones((h, pitch), device="cuda")
    tgt = A.ec_target()
    for pvp in (None, (2, 3, w, h)):
        assert A.marshal().target(color, buf[:, :w], pvp, 0, C.addressof(tgt)) and tgt.depth == buf.data_ptr()
        for bad in (buf[:h - 1, :w], buf[:0, :w], buf[:, :w - 1], buf.reshape(-1)):
            assert not A.marshal().target(color, bad, pvp, 0, C.addressof(tgt))
            with pytest.raises(ValueError):
                api._target(color, bad, pvp, 0)
    assert A.marshal().target(color, buf[:4, :5], (0, 0, 5, 4), 0, C.addressof(tgt))
    assert not A.marshal().target(color, buf[:4, :5], (0, 0, 5, 5), 0, C.addressof(tgt))


def test_calls_with_a_short_output_depth_are_refused():
    require_gpu()
    h, w = 20, 36
    color = torch.zeros((h, w), dtype=torch.int32, device="cuda").view(torch.uint32)
    depth = torch.full((h, w), 0.5, device="cuda")
    images = [ec.Image(color, depth)] * 2
    out = torch.zeros((h, w), dtype=torch.int32, device="cuda").view(torch.uint32)
    for bad in (torch.ones((h, w), device="cuda")[:h - 1], torch.ones((h, w), device="cuda")[:, :w - 1]):
        with pytest.raises(ValueError):
            ec.composite_depth(images, out, bad)
        with pytest.raises(ValueError):
            ec.Batch([ec.Job("depth", images, out, bad)], config={})
        with pytest.raises(ValueError):
            ec.Schedule("depth", "binary_swap", images, out, bad)
