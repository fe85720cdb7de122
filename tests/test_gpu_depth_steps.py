"""The depth merge gives the same bits whichever way its lanes take their pixels:
with any number of unaligned inputs among aligned ones."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu


def _merge(images, w, h):
    c, d = torch.full((h, w), 7, dtype=torch.int32, device="cuda"), torch.full((h, w), 7.0, device="cuda")
    win = torch.full((h, w), 7, dtype=torch.int16, device="cuda")
    ec.composite_depth(images, c.view(torch.uint32), d, winner=win)
    ec.default_context().check_status()
    return c, d, win


def _inputs(n, single, w, h, rect, g):
    """n inputs of which the first `single` lie in rows of any alignment; returns
    them and aligned copies."""
    x, y, iw, ih = rect
    a, b = [], []
    for k in range(n):
        c = torch.randint(-(1 << 31), 1 << 31, (ih, iw), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
        d = torch.randint(0, 12, (ih, iw), generator=g, device="cuda").float() / 10        # ties, and depths of 1 and more
        pitch = (iw + 3) // 4 * 4
        cc, dd = torch.zeros((ih, pitch), dtype=torch.int32, device="cuda"), torch.ones((ih, pitch), device="cuda")
        cc[:, :iw], dd[:, :iw] = c, d
        whole = ec.Image(cc[:, :iw].view(torch.uint32), dd[:, :iw], rect, rect)
        b.append(whole)
        if k < single:
            c1, d1 = torch.zeros((ih, iw + 1), dtype=torch.int32, device="cuda"), torch.ones((ih, iw + 1), device="cuda")
            c1[:, 1:], d1[:, 1:] = c, d
            a.append(ec.Image(c1[:, 1:].view(torch.uint32), d1[:, 1:], rect, rect))
        else:
            a.append(whole)
    return a, b


@pytest.mark.parametrize("n", [1, 2, 5, 17])
@pytest.mark.parametrize("w,h,rect", [(1, 1, (0, 0, 1, 1)), (131, 9, (0, 0, 131, 9)), (260, 33, (4, 3, 253, 27))])
def test_any_share_of_unaligned_inputs(w, h, rect, n):
    require_gpu()
    g = torch.Generator(device="cuda")
    g.manual_seed(w + n)
    for single in sorted({0, 1, n // 2, n // 2 + 1, n} & set(range(n + 1))):
        a, b = _inputs(n, single, w, h, rect, g)
        assert all(torch.equal(p, q) for p, q in zip(_merge(a, w, h), _merge(b, w, h))), single
