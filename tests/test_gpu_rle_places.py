"""GPU parity of where a batch's chunks are placed: images whose first and last
chunks fall on every position of the groups of 32 chunks whose sizes are summed
while they are coded, empty ones between them, with flat, few-run and dense
chunks side by side, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu
CHUNK = ec.EC_RLE_CHUNK


def _image(r, chunks):
    """`chunks` chunks (the last one cut short), each flat, of a few runs or dense."""
    img = np.zeros((chunks, CHUNK), np.uint32)
    for row in img:
        k = int(r.integers(0, 4))
        if k == 0:
            row[:] = r.integers(0, 1 << 32, size=CHUNK, dtype=np.uint64)
        elif k == 1:
            row[: int(r.integers(1, 200))] = r.integers(0, 1 << 32, dtype=np.uint64)
    return img.reshape(1, -1)[:, : max(0, chunks * CHUNK - int(r.integers(0, 40)))]


@pytest.mark.parametrize("counts", [[1], [33], [1] * 70, [31, 1, 0, 33, 32, 64, 65], [0, 0, 5, 0], [100, 0, 28, 200, 3],
                                    [1, 30, 1] * 10 + [0], [700, 9]])
def test_places_match_the_oracle(counts):
    require_gpu()
    r = np.random.default_rng(len(counts) * 1000 + sum(counts))
    images = [_image(r, n) for n in counts]
    modes = [1 + int(r.integers(0, 2)) for _ in counts]
    jobs = [(torch.from_numpy(a.view(np.int32)).cuda().view(torch.uint32), m, None, None, None)
            for a, m in zip(images, modes)]
    outs = ec.rle_compress_batch(jobs)
    ec.default_context().check_status()
    for (dst, size), a, m in zip(outs, images, modes):
        want = oracle.rle_compress(a, m)
        assert int(size.item()) == len(want)
        assert dst[: len(want)].cpu().numpy().tobytes() == want
