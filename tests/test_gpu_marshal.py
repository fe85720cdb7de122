"""The native argument marshalling fills the same descriptors as the binding's
own checks for every form it takes, and leaves the others to them."""
import ctypes as C

import numpy as np
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu
from paper_1902_08755_gb300 import _abi as A
from paper_1902_08755_gb300 import api

pytestmark = pytest.mark.gpu


class Sub(torch.Tensor):
    pass


def _forms():
    z = dict(device="cuda")
    u8 = torch.zeros((20, 36), dtype=torch.int32, **z)
    f32, f16 = torch.zeros((20, 36, 4), **z), torch.zeros((20, 36, 4), dtype=torch.float16, **z)
    d = torch.ones((20, 36), **z)
    yield "plain", ec.Image(u8, d, (3, 4, 36, 20), (5, 6, 7, 8)), True
    yield "lists", ec.Image(u8.view(torch.uint32), d, [3, 4, 30, 20], [5, 6, 7, 8]), True
    yield "no rects", ec.Image(f32), True
    yield "half, cropped", ec.Image(f16[2:9, 3:30], None, (0, -5, 27, 7)), True
    yield "cropped with depth", ec.Image(u8[2:9, 3:30], d[2:9, 3:30], None, (1, 1, 2, 2)), True
    yield "empty", ec.Image(f32[:0]), True
    yield "numpy ints", ec.Image(u8, d, tuple(np.arange(4)), (0, 0, 1, 1)), False
    yield "float rect", ec.Image(f32, None, (0.0, 0, 36, 20)), False
    yield "array rect", ec.Image(f32, None, np.array([0, 0, 36, 20])), False
    yield "bool in rect", ec.Image(f32, None, (False, 0, 36, 20)), False
    yield "subclass", ec.Image(f32.as_subclass(Sub)), False
    yield "parameter", ec.Image(torch.nn.Parameter(f32.clone())), None
    yield "transposed", ec.Image(u8.t()), False
    yield "three channels", ec.Image(f32[..., :3]), False
    yield "double", ec.Image(f32.double()), False
    yield "on the host", ec.Image(u8.cpu(), d.cpu()), False
    yield "pvp too large", ec.Image(u8, d, (0, 0, 37, 20)), False
    yield "other depth pitch", ec.Image(u8[:, :30], torch.ones((20, 30), **z)), False
    yield "half depth", ec.Image(u8, d.half()), False
    yield "short depth", ec.Image(u8, d[:19]), False


@pytest.mark.parametrize("need", [api._NO_DEPTH, api._DEPTH, api._ANY_DEPTH])
def test_images(need):
    require_gpu()
    for name, im, taken in _forms():
        depth = need == api._DEPTH or (need == api._ANY_DEPTH and im.depth is not None)
        arr = (A.ec_image * 2)()
        got = A.marshal().images([im, im], 0, need, C.addressof(arr))
        try:
            want = api._image_struct(im, 0, depth)
        except (ValueError, TypeError, RuntimeError):
            want = None
        if want is None:
            assert not got, name
            with pytest.raises((ValueError, TypeError, RuntimeError)):
                api._images([im], 0, need)
            continue
        if taken is False and not (not depth and "depth" in name):
            assert not got, name                       # (a rarer form: the binding's checks take it)
        if got:
            assert bytes(arr[0]) == bytes(want) and bytes(arr[1]) == bytes(want), name
        else:
            assert taken is not True, name
        assert bytes(api._images([im], 0, need)[0]) == bytes(want), name


def test_targets_orders_and_gradients():
    require_gpu()
    f = torch.zeros((9, 17, 4), device="cuda")
    tgt = A.ec_target()
    assert A.marshal().target(f, None, (1, 2, 16, 9), 0, C.addressof(tgt))
    assert (tgt.pvp.tup(), tgt.pitch, tgt.format, tgt.color, tgt.depth) == ((1, 2, 16, 9), 17, A.EC_RGBA32F,
                                                                           f.data_ptr(), None)
    for bad in ((f, None, (0, 0, 18, 9)), (f.cpu(), None, None), (f, f, None), (f.double(), None, None)):
        assert not A.marshal().target(*bad, 0, C.addressof(tgt))
    with pytest.raises(ValueError):
        api._target(f, None, (0, 0, 18, 9), 0)
    assert list(api._order((2, 0, 1), 3)) == [2, 0, 1] and list(api._order(np.array([1, 0]), 2)) == [1, 0]
    with pytest.raises(ValueError):
        api._order([0, 1], 3)
    layers = [ec.Image(f), ec.Image(f)]
    g = [torch.zeros_like(f), torch.zeros_like(f).half()]
    fmt, ptrs = api._gradients(g[:1] * 2, layers, 0)
    assert fmt == A.EC_RGBA32F and list(ptrs) == [g[0].data_ptr()] * 2
    assert api._gradients(g[1:] * 2, layers, 0)[0] == A.EC_RGBA16F
    for bad in (g, g[:1], [g[0], g[0][:8]], [g[0], g[0].cpu()], [g[0], torch.zeros((9, 17), device="cuda", dtype=torch.int32)]):
        with pytest.raises(ValueError):
            api._gradients(bad, layers, 0)
