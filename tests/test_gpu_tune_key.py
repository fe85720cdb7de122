"""The tune cache tells batches apart whose items run in different kernels, and
knows a batch again whose items run in the same ones."""
import pytest
import torch

import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu


def _plan(mode, shift, dx):
    """Two inputs of 40 x 24, stored `shift` pixels into rows of 64, `dx` columns
    into an output of 60 x 24."""
    w, h = 40, 24
    images = []
    for _ in range(2):
        if mode == "depth":
            c = torch.zeros((h, 64), dtype=torch.int32, device="cuda")[:, shift:shift + w]
            images.append(ec.Image(c.view(torch.uint32), torch.ones((h, 64), device="cuda")[:, shift:shift + w], (dx, 0, w, h)))
        else:
            images.append(ec.Image(torch.zeros((h, 64, 4), dtype=torch.float16, device="cuda")[:, shift:shift + w], None,
                                   (dx, 0, w, h)))
    if mode == "depth":
        job = ec.Job("depth", images, torch.zeros((h, 60), dtype=torch.int32, device="cuda").view(torch.uint32),
                     torch.zeros((h, 60), device="cuda"))
    else:
        job = ec.Job("alpha", images, torch.zeros((h, 60, 4), dtype=torch.float16, device="cuda"))
    plan = ec.Batch([job])
    plan.run()
    torch.cuda.synchronize()
    plan.close()


@pytest.mark.parametrize("mode", ["depth", "alpha"])
def test_keys_follow_alignment_and_place(mode, tmp_path, monkeypatch):
    require_gpu()
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("EC_AUTOTUNE_CACHE", str(cache))
    for shift, dx in [(0, 0), (1, 0), (0, 20)]:          # aligned; rows of any alignment; elsewhere in the output
        _plan(mode, shift, dx)
    keys = [line.split()[0] for line in cache.read_text().splitlines()]
    assert len(keys) == 3 and len(set(keys)) == 3
    _plan(mode, 0, 0)                                    # other buffers, the same layout
    assert len(cache.read_text().splitlines()) == 3
