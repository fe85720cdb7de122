"""Jobs without inputs, or whose inputs all lie elsewhere, write the background
of their whole output: the colour and depth that a single call without inputs
writes, and no winner."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu


def _outs(kind, w, h):
    z = dict(device="cuda")
    if kind == "depth":
        c = torch.full((h, w), 7, dtype=torch.int32, **z)
    else:
        c = torch.full((h, w, 4), 7.0, dtype=torch.float16 if kind == "half" else torch.float32, **z)
    return c, torch.full((h, w), 7.0, **z), torch.full((h, w), 7, dtype=torch.int16, **z)


def _elsewhere(kind, w):
    z = dict(device="cuda")
    at = (w + 3, 0, 8, 8)
    if kind == "depth":
        return [ec.Image(torch.full((8, 8), 3, dtype=torch.int32, **z).view(torch.uint32), torch.zeros((8, 8), **z), at)]
    if kind == "depth32":
        return [ec.Image(torch.ones((8, 8, 4), **z), torch.zeros((8, 8), **z), at)]
    return [ec.Image(torch.ones((8, 8, 4), dtype=torch.float16 if kind == "half" else torch.float32, **z), None, at)]


@pytest.mark.parametrize("elsewhere", [False, True])
@pytest.mark.parametrize("w,h", [(1, 1), (5, 3), (131, 17)])
def test_jobs_without_inputs_write_the_background(w, h, elsewhere):
    require_gpu()
    jobs, outs = [], []
    for kind in ("depth", "depth32", "half", "float"):
        images = _elsewhere(kind, w) if elsewhere else []
        c, d, win = _outs(kind, w, h)
        one = _outs(kind, w, h)
        cv = c.view(torch.uint32) if kind == "depth" else c
        ov = one[0].view(torch.uint32) if kind == "depth" else one[0]
        if kind.startswith("depth"):
            jobs.append(ec.Job("depth", images, cv, d, winner=win))
            ec.composite_depth(images, ov, one[1], winner=one[2])
        else:
            jobs.append(ec.Job("alpha", images, cv, t_final=d))
            ec.composite_alpha(images, ov, t_final=one[1])
        outs.append((kind, (c, d, win), one))
    plan = ec.Batch(jobs, config={})
    plan.run()
    ec.default_context().check_status()
    for kind, (c, d, win), one in outs:
        assert not c.any() and bool((d == 1).all()), kind
        assert not one[0].any() and bool((one[1] == 1).all()), kind
        if kind.startswith("depth"):
            assert bool((win == -1).all()) and bool((one[2] == -1).all()), kind
    plan.close()
