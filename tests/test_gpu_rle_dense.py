"""GPU parity of the codec on chunks of many tokens: streams whose tokens fall on
every edge of the decoder's 64-byte windows and 128-byte lines, streams around
the size that picks the decoder's path, images of odd width stored in one run,
and malformed streams of many tokens, all against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1902_08755_gb300 as ec
from ec_testutil import np_of, require_gpu

pytestmark = pytest.mark.gpu
CHUNK = ec.EC_RLE_CHUNK


def _dev(buf: bytes) -> torch.Tensor:
    return torch.from_numpy(np.frombuffer(buf, np.uint8).copy()).cuda()


def _plane_stream(r, n, kind):
    """Random valid tokens that decode to n bytes (any split, also ones no
    encoder makes: repeats of one byte, literal tokens in a row)."""
    out = bytearray()
    while n > 0:
        k = kind if kind != "mixed" else r.choice(["short", "literal", "repeat", "long"])
        if k == "repeat" or (k in ("short", "long") and r.random() < 0.6):
            m = int(min(n, r.integers(1, 129 if k != "short" else 6)))
            out += bytes([127 + m, int(r.integers(0, 256))])
        else:
            m = int(min(n, r.integers(1, 6) if k == "short" else r.choice([1, 2, 31, 61, 62, 63, 64, 125, 126, 127, 128])))
            out += bytes([m - 1]) + r.integers(0, 256, size=m, dtype=np.uint8).tobytes()
        n -= m
    return bytes(out)


def _container(r, w, h, mode, kinds):
    n = w * h
    head = oracle.rle_compress(np.zeros((h, w), np.uint32), mode)[:32]
    ends, pay = [], bytearray()
    for c0 in range(0, n, CHUNK):
        for p in range(4):
            pay += _plane_stream(r, min(CHUNK, n - c0), kinds[p])
            ends.append(len(pay))
    return bytes(head) + np.array(ends, np.uint32).tobytes() + bytes(pay)


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("w,h", [(4096, 2), (4095, 1), (1, 65), (997, 9), (64, 200), (2050, 3)])
@pytest.mark.parametrize("kinds", [("mixed",) * 4, ("short",) * 4, ("literal", "short", "long", "repeat"),
                                   ("repeat", "repeat", "literal", "repeat")])
def test_decoder_takes_any_valid_tokens(w, h, mode, kinds):
    require_gpu()
    r = np.random.default_rng([w, h, mode, len(kinds[0])])
    buf = _container(r, w, h, mode, kinds)
    if oracle.rle_decompress_status(buf, w, h) != 0:
        # longer than the all-literal coding: refused by both
        ec.rle_decompress(_dev(buf), w, h)
        assert ec.default_context().status_sync() == 4
        return
    want = oracle.rle_decompress(buf, w, h)
    for pitch in (w, w + 3):
        dst = torch.full((h, pitch), 0x5A5A5A5A, dtype=torch.int32, device="cuda").view(torch.uint32)
        ec.rle_decompress(_dev(buf), w, h, dst=dst)
        ec.default_context().check_status()
        got = np_of(dst)
        assert np.array_equal(got[:, :w], want)
        assert (got[:, w:].view(np.int32) == 0x5A5A5A5A).all()


@pytest.mark.parametrize("seed", range(24))
def test_malformed_streams_of_many_tokens(seed):
    require_gpu()
    r = np.random.default_rng(1000 + seed)
    w, h = int(r.integers(500, 1500)), int(r.integers(4, 9))
    img = r.integers(0, 1 << 32, size=(h, w), dtype=np.uint64).astype(np.uint32)
    img[:, : w // 3] &= np.uint32(0xFF00FF00)
    buf = bytearray(oracle.rle_compress(img, 1 + seed % 2))
    tab = 32 + 16 * (-(-w * h // CHUNK))
    for _ in range(1 + seed % 5):
        i = int(r.integers(tab, len(buf)))
        buf[i] ^= 1 << int(r.integers(0, 8))
    out = ec.rle_decompress(_dev(bytes(buf)), w, h)
    st = ec.default_context().status_sync()
    assert st == oracle.rle_decompress_status(bytes(buf), w, h)
    if st == 0:
        assert np.array_equal(np_of(out), oracle.rle_decompress(bytes(buf), w, h))
