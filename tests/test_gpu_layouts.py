"""The paths that follow from an input's layout and a launch's size give the same
bits as the general ones: inputs whose rows are not 16-byte groups against
aligned copies of them, batches of covered, partly covered and clipped tiles
against one call per job, and gradients of frames and stacks whose rows per CTA
differ against the oracle."""
import numpy as np
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu
from test_gpu_grad import _bwd_case, _check_against_oracle, _run_bwd

pytestmark = pytest.mark.gpu


def _same(a, b):
    if a.dtype == torch.uint32:
        a, b = a.view(torch.int32), b.view(torch.int32)
    return torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


def _stored(shape, dtype, pitch, shift, g):
    """Random rows of `pitch` pixels whose first pixel lies `shift` pixels into the
    allocation."""
    h, w = shape[:2]
    tail = shape[2:]
    per = int(np.prod(tail)) if tail else 1
    buf = torch.zeros((shift + h * pitch) * per, dtype=dtype, device="cuda")
    v = buf[shift * per:].view(h, pitch, *tail)
    if dtype == torch.int32:
        v.copy_(torch.randint(-(1 << 31), 1 << 31, v.shape, generator=g, device="cuda", dtype=torch.int64))
    else:
        v.copy_(torch.rand(v.shape, generator=g, device="cuda"))
    return v[:, :w]


def _sources(n, w, h, kind, odd, g, inside):
    """n images of about w x h, with odd rows or rows of 16-byte groups."""
    r = np.random.default_rng([n, w, h, odd])
    out = []
    for k in range(n):
        iw, ih = (w, h) if inside else (int(r.integers(1, w + 1)), int(r.integers(1, h + 1)))
        x, y = (0, 0) if inside else (int(r.integers(0, w - iw + 1)), int(r.integers(0, h - ih + 1)))
        pitch, shift = (iw + 1 + 2 * k % 4 | 1, k % 3) if odd else ((iw + 7) // 4 * 4, 0)
        if not odd:
            x = x // 4 * 4
        pvp = (x, y, iw, ih)
        roi = pvp if inside or k % 3 else (x, y, max(1, iw - 2), max(1, ih - 1))
        if kind == "depth":
            c, d = _stored((ih, iw), torch.int32, pitch, shift, g), _stored((ih, iw), torch.float32, pitch, shift, g)
            out.append(ec.Image(c.view(torch.uint32), d, pvp, roi))
        elif kind == "depth32":
            out.append(ec.Image(_stored((ih, iw, 4), torch.float32, pitch, 0, g),
                                _stored((ih, iw), torch.float32, pitch, shift, g), pvp, roi))
        else:
            dt = torch.float16 if kind == "half" else torch.float32
            out.append(ec.Image(_stored((ih, iw, 4), dt, pitch, shift, g), None, pvp, roi))
    return out


def _aligned(im):
    """The same image stored in rows of whole 16-byte groups, from a multiple of four on."""
    h, w = im.color.shape[:2]
    px, py, pw, ph = im.pvp
    lead = px % 4
    pitch = (lead + w + 3) // 4 * 4
    c = torch.zeros((h, pitch, *im.color.shape[2:]), dtype=torch.int32 if im.color.dtype == torch.uint32 else im.color.dtype,
                    device="cuda")
    c[:, lead:lead + w] = im.color.view(torch.int32) if im.color.dtype == torch.uint32 else im.color
    d = None
    if im.depth is not None:
        d = torch.ones((h, pitch), device="cuda")
        d[:, lead:lead + w] = im.depth
    return ec.Image(c.view(torch.uint32) if im.color.dtype == torch.uint32 else c, d, (px - lead, py, pitch, h), im.roi)


def _targets(kind, w, h):
    if kind == "depth":
        return (torch.full((h, w), 7, dtype=torch.int32, device="cuda").view(torch.uint32),
                torch.full((h, w), 7.0, device="cuda"), torch.full((h, w), 7, dtype=torch.int16, device="cuda"))
    dt = torch.float16 if kind == "half" else torch.float32
    return (torch.full((h, w, 4), 7.0, dtype=dt, device="cuda"), torch.full((h, w), 7.0, device="cuda"),
            torch.full((h, w), 7, dtype=torch.int16, device="cuda"))


def _run(kind, images, w, h):
    c, d, win = _targets(kind, w, h)
    if kind.startswith("depth"):
        ec.composite_depth(images, c, d, winner=win)
        return c, d, win
    ec.composite_alpha(images, c, t_final=d)
    return c, d


@pytest.mark.parametrize("kind", ["depth", "depth32", "half", "float"])
@pytest.mark.parametrize("w,h,n", [(1, 1, 1), (127, 5, 3), (128, 4, 4), (129, 9, 5), (333, 17, 9), (515, 8, 17)])
def test_unaligned_rows_equal_aligned_ones(kind, w, h, n):
    require_gpu()
    g = torch.Generator(device="cuda")
    g.manual_seed(w * 1000 + n)
    images = _sources(n, w, h, kind, True, g, False)
    got = _run(kind, images, w, h)
    want = _run(kind, [_aligned(im) for im in images], w, h)
    ec.default_context().check_status()
    assert all(_same(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("config", [{}, dict(depth_tile_h=4, alpha32_tile_h=16, alpha16_tile_h=32, ctas_per_sm=1)])
def test_batch_kinds_equal_single_calls(config):
    """Every kind of job, with rows of both kinds, covered by its inputs or not, of
    sizes at the edges of a tile; fewer items than CTAs and many more."""
    require_gpu()
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    jobs, want = [], []
    for w, h, n in [(1, 1, 1), (31, 8, 2), (32, 9, 8), (127, 16, 9), (128, 8, 4), (129, 31, 5), (256, 33, 33), (700, 300, 3),
                    (5, 3, 0)]:
        for kind in ("depth", "depth32", "half", "float"):
            for odd in (False, True):
                for inside in (True, False):
                    images = _sources(n, w, h, kind, odd, g, inside)
                    c, d, win = _targets(kind, w, h)
                    if kind.startswith("depth"):
                        jobs.append(ec.Job("depth", images, c, d, winner=win))
                        want.append(_run(kind, images, w, h) if n else None)
                    else:
                        jobs.append(ec.Job("alpha", images, c, t_final=d))
                        want.append(_run(kind, images, w, h) if n else None)
    plan = ec.Batch(jobs, config=config)
    for _ in range(2):
        plan.run()
        ec.default_context().check_status()
        for jb, ref in zip(jobs, want):
            got = (jb.out_color, jb.out_depth, jb.winner) if jb.mode == "depth" else (jb.out_color, jb.t_final)
            if ref is not None:
                assert all(_same(a, b) for a, b in zip(got, ref)), (jb.mode, jb.out_color.shape, len(jb.images))
    plan.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("n,w,h", [(1, 32, 1), (3, 33, 2), (12, 70, 200), (65, 40, 130), (128, 33, 70)])
def test_rows_per_cta_follow_the_oracle(n, w, h, dtype):
    require_gpu()
    oimgs, gimgs, order, out_pvp, grad = _bwd_case(90 + n, dtype, n=n, W=w, H=h)
    grads = _run_bwd(gimgs, order, out_pvp, grad, torch.float32)
    _check_against_oracle(oimgs, grads, order, out_pvp, grad, torch.float32)
