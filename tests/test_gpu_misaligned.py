"""Float images whose buffers start at any multiple of their channel size (a view
into a packed buffer): assembly and depth merge give the same bits as with
aligned copies, whichever of the buffers it is."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu
G = 7.0                                                # guard value around every view


def _view(t, off, pitch=None):
    """A copy of the [h][w][4] image whose first channel lies `off` channels into
    its allocation; returns (view, whole allocation)."""
    h, w = t.shape[:2]
    pitch = pitch or w
    buf = torch.full((off + h * pitch * 4 + 8,), G, dtype=t.dtype, device="cuda")
    v = buf[off:off + h * pitch * 4].view(h, pitch, 4)[:, :w]
    v.copy_(t)
    return v, buf


def _rand(h, w, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand((h, w, 4), generator=g, device="cuda").to(dtype)


def _places(w, h):
    """Three overlapping rectangles and one pixel."""
    return [(0, 0, max(1, w * 2 // 3), h), (w // 3, h // 4, w - w // 3, h - h // 4), (0, 0, w, max(1, h // 2)), (w - 1, h - 1, 1, 1)]


def _run(call, w, h, dtype, soff, doff, pitch):
    out, buf = _view(torch.zeros((h, w, 4), dtype=dtype, device="cuda"), doff, pitch)
    rects = _places(w, h)
    if call == "pixels":
        owned = [((w + 1) // 2, (h + 1) // 2), (w // 2, (h + 1) // 2), ((w + 1) // 2, h // 2), (w // 2, h // 2)]
        offs = [(0, 0), (1, 0), (0, 1), (1, 1)]
        keep = [(o, _view(_rand(oh, ow, dtype, i), soff)[0]) for i, ((ow, oh), o) in enumerate(zip(owned, offs)) if ow and oh]
        ec.assemble_pixels([t for _, t in keep], [o for o, _ in keep], (2, 2), out)
    else:
        images = [_view(_rand(r[3], r[2], dtype, 10 + i), soff, r[2] + i % 2)[0] for i, r in enumerate(rects)]
        if call == "depth":
            depth, win = torch.zeros((h, pitch), device="cuda")[:, :w], torch.zeros((h, w), dtype=torch.int16, device="cuda")
            g = torch.Generator(device="cuda")
            g.manual_seed(20)
            ims = [ec.Image(t, torch.rand((r[3], r[2] + i % 2), generator=g, device="cuda")[:, :r[2]], r, r)
                   for i, (t, r) in enumerate(zip(images, rects))]
            ec.composite_depth(ims, out, depth, winner=win)
        else:
            ims = [ec.Image(t, None, r, r) for t, r in zip(images, rects)]
            (ec.average if call == "average" else ec.assemble_tiles)(ims, out)
    ec.default_context().check_status()
    # nothing before, after or between the rows
    assert bool((buf[:doff] == G).all()) and bool((buf[doff + h * pitch * 4:] == G).all())
    assert bool((buf[doff:doff + h * pitch * 4].view(h, pitch, 4)[:, w:] == G).all())
    return (out.clone(), depth.clone(), win) if call == "depth" else (out.clone(),)


@pytest.mark.parametrize("call,dtype", [("tiles", torch.float32), ("tiles", torch.float16), ("average", torch.float32),
                                        ("average", torch.float16), ("pixels", torch.float32), ("pixels", torch.float16),
                                        ("depth", torch.float32)])
@pytest.mark.parametrize("w,h", [(1, 1), (33, 9), (130, 41)])
def test_buffers_at_any_channel(call, dtype, w, h):
    require_gpu()
    for pitch in (w, w + 1):
        want = _run(call, w, h, dtype, 0, 0, pitch)
        for soff, doff in ([(1, 0), (2, 0), (0, 1), (3, 2)] if dtype == torch.float32 else [(2, 0), (0, 2), (2, 6)]):
            got = _run(call, w, h, dtype, soff, doff, pitch)
            assert all(torch.equal(a, b) for a, b in zip(got, want)), (soff, doff, pitch)


def test_more_inputs_than_the_small_instances_hold():
    """70 tiles, one of them misaligned."""
    require_gpu()
    h, w = 24, 70
    outs = []
    for off in (0, 1):
        images = [ec.Image(_view(_rand(h, 1, torch.float32, i), off if i == 33 else 0)[0], None, (i, 0, 1, h), (i, 0, 1, h))
                  for i in range(w)]
        out = torch.zeros((h, w, 4), device="cuda")
        ec.assemble_tiles(images, out)
        outs.append(out)
    ec.default_context().check_status()
    assert torch.equal(outs[0], outs[1]) and bool((outs[0] != 0).any())
