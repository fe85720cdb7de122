"""A launch that the CUDA runtime refuses is reported by the call that made it
and leaves nothing behind: the next call, of this library or of another, is not
failed by it."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu


def test_a_refused_launch_leaves_no_error_behind():
    require_gpu()
    h = 4 * 65535 + 1                                 # one row of CTAs more than a grid takes
    color = torch.zeros((h, 1), dtype=torch.int32, device="cuda").view(torch.uint32)
    depth = torch.full((h, 1), 0.5, device="cuda")
    out, od = torch.zeros((h, 1), dtype=torch.int32, device="cuda"), torch.zeros((h, 1), device="cuda")
    small = [ec.Image(torch.full((8, 8), 5, dtype=torch.int32, device="cuda").view(torch.uint32),
                      torch.full((8, 8), 0.25, device="cuda"))]
    oc, o2 = torch.zeros((8, 8), dtype=torch.int32, device="cuda"), torch.zeros((8, 8), device="cuda")

    def refused():
        with pytest.raises(ec.EcError):
            ec.composite_depth([ec.Image(color, depth)], out.view(torch.uint32), od)
    refused()
    assert torch.equal(torch.arange(5, device="cuda") + 1, torch.arange(1, 6, device="cuda"))
    refused()
    plan = ec.Batch([ec.Job("depth", small, oc.view(torch.uint32), o2)], config={})
    refused()
    plan.run()
    torch.cuda.synchronize()
    assert bool((oc == 5).all()) and bool((o2 == 0.25).all())
    plan.close()
    assert not out.any() and not od.any()
