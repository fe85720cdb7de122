"""GPU parity of the compressor where chunks find its scratch pool full, counted
from the streams themselves: the allocation-free entry point's pool has room for
512 bytes per chunk of its largest image and little more, and the images here
need more, in chunks of few runs, of many, and of both.  Those that find it full
are coded again when placed."""
import numpy as np
import pytest
import torch

import oracle
import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu
from paper_1902_08755_gb300 import _abi as A

pytestmark = pytest.mark.gpu
CHUNK = ec.EC_RLE_CHUNK
CHUNKS = A.EC_RLE_NOALLOC_MAX_CHUNKS
SCRATCH = 256 + 537 * CHUNKS                       # EC_RLE_NOALLOC_SCRATCH_BYTES


def _image(kind, seed):
    """One row per chunk.  "sparse": 126 noisy elements, then one value (127 change
    points in every plane, 127 units or fewer in mode 0), as few-run chunks may
    have at most; "mixed": every fifth noise, every fifth flat."""
    r = np.random.default_rng(seed)
    rows = 512
    img = np.repeat(r.integers(0, 1 << 32, size=(rows, 1), dtype=np.uint64).astype(np.uint32), CHUNK, axis=1)
    img[:, :126] = r.integers(0, 1 << 32, size=(rows, 126), dtype=np.uint64)
    if kind == "mixed":
        img[2::5] = r.integers(0, 1 << 32, size=img[2::5].shape, dtype=np.uint64)
        img[4::5] = 7
    return np.tile(img, (CHUNKS // rows, 1))


def _chunk_sizes(stream, mode):
    per = 1 if mode == 0 else 4
    ends = np.frombuffer(stream, np.uint32, per * CHUNKS, 32).astype(np.int64)
    return np.diff(ends[per - 1::per], prepend=0)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("kind", ["sparse", "mixed"])
def test_chunks_that_find_the_pool_full(kind, mode):
    require_gpu()
    img = _image(kind, [7, mode, kind == "mixed"])
    want = oracle.rle_compress(img, mode)
    sizes = _chunk_sizes(want, mode)
    # every few-run chunk is larger than a chunk's slot, and all chunks together
    # than the whole scratch: most of them find the pool full
    few = np.isin(np.arange(CHUNKS) % 512 % 5, [0, 1, 3]) | (kind == "sparse")
    assert (sizes[few] > 512).all() and sizes.sum() > SCRATCH
    h, w = img.shape
    src = torch.from_numpy(img.view(np.int32)).cuda()
    dst = torch.zeros(ec.rle_max_size(w, h), dtype=torch.uint8, device="cuda")
    size, st = torch.zeros(1, dtype=torch.uint64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        dst.zero_()
        A.check(A.load().ec_rle_compress_noalloc(src.data_ptr(), w, h, w, mode, dst.data_ptr(), dst.numel(),
                                                 size.data_ptr(), st.data_ptr(), torch.cuda.current_stream().cuda_stream),
                "noalloc")
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        assert int(size.item()) == len(want)
        assert dst[:len(want)].cpu().numpy().tobytes() == want
