"""FP16 layers in rows that are not 16-byte groups, read as whole pixels or by
halves, in one call alone or together, blend to the same bits as aligned copies;
single calls and batches."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu


def _layer(t, off, pitch):
    """A copy of [h][w][4] whose first half lies `off` halves into its allocation."""
    h, w = t.shape[:2]
    buf = torch.full((off + h * pitch * 4 + 8,), 9.0, dtype=torch.float16, device="cuda")
    v = buf[off:off + h * pitch * 4].view(h, pitch, 4)[:, :w]
    v.copy_(t)
    return v


def _out(w, h, off):
    return _layer(torch.zeros((h, w, 4), dtype=torch.float16, device="cuda"), off, w), torch.zeros((h, w), device="cuda")


# per layer in turn: halves before the first pixel (multiples of 4: whole pixels)
@pytest.mark.parametrize("offs", [(0,), (4, 12), (1,), (2, 3), (0, 4, 1, 6)])
@pytest.mark.parametrize("w,h,n", [(1, 1, 1), (63, 9, 3), (65, 17, 8), (130, 25, 17), (64, 8, 66)])
def test_reads_equal_aligned_ones(w, h, n, offs):
    require_gpu()
    g = torch.Generator(device="cuda")
    g.manual_seed(w * n + len(offs))
    aligned, odd = [], []
    for k in range(n):
        x, y = (0, 0) if k % 2 else (k % w, k % h)           # every other layer covers the frame
        a = torch.rand((h - y, w - x, 1), generator=g, device="cuda") * 0.5
        t = torch.cat([torch.rand((h - y, w - x, 3), generator=g, device="cuda") * a, a], 2).half()
        roi = (x, y, w - x, h - y)
        aligned.append(ec.Image(_layer(t, 0, w - x + (w - x) % 2), None, roi, roi))
        odd.append(ec.Image(_layer(t, offs[k % len(offs)], (w - x) | 1), None, roi, roi))
    want, left = _out(w, h, 0)
    ec.composite_alpha(aligned, want, t_final=left)
    for off in (0, offs[-1]):
        got, gleft = _out(w, h, off)
        ec.composite_alpha(odd, got, t_final=gleft)
        assert torch.equal(got, want) and torch.equal(gleft, left)
        got, gleft = _out(w, h, off)
        plan = ec.Batch([ec.Job("alpha", odd, got, t_final=gleft)], config={})
        plan.run()
        ec.default_context().check_status()
        assert torch.equal(got, want) and torch.equal(gleft, left)
        plan.close()
