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


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("m", [33, 64, 97, 128])
@pytest.mark.parametrize("w,h", [(CHUNK, 2), (1001, 9)])
def test_chunks_of_many_runs_without_short_ones(m, w, h, mode):
    """Chunks of 33 to 128 change points (the list's whole range above the
    few-run case) whose runs all have three or more elements, so every plane is
    repeat tokens only: runs of 3, of whole tokens, of one more, and long ones."""
    require_gpu()
    r = np.random.default_rng([m, w, mode])
    n = w * h
    flat = np.zeros(n, np.uint32)
    for c0 in range(0, n, CHUNK):
        left = min(CHUNK, n - c0)
        k = min(m, left // 3)
        L = np.full(k, 3)
        for j, want in zip(r.permutation(k), [125, 126, 253, 0, 1, 254, 60]):     # 128, 129, 256, 3, 4, 257, 63
            if L.sum() + want <= left:
                L[j] += want
        L[int(r.integers(0, k))] += left - L.sum()
        e = r.integers(0, 1 << 32, size=k, dtype=np.uint64).astype(np.uint32)
        flat[c0:c0 + left] = np.repeat(e, L)
    img = flat.reshape(h, w)
    want = oracle.rle_compress(img, mode)
    buf, size = ec.rle_compress(torch.from_numpy(img.view(np.int32)).cuda().view(torch.uint32), mode)
    ec.default_context().check_status()
    assert buf[: int(size.item())].cpu().numpy().tobytes() == want
