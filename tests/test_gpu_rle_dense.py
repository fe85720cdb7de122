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


def _mixed(kind, w, h, seed):
    """Rows that take each path of the compressor: flat, a few runs, runs of one
    to three bytes in a plane, more change points than a list holds, noise."""
    r = np.random.default_rng(seed)
    img = np.zeros((h, w), np.uint32)
    flat = img.reshape(-1)
    n = flat.size
    if kind == "edges":                              # changes at every edge of groups, warps and chunks
        for q in [0, 1, 3, 4, 127, 128, 511, 512, 1023, 1024, 1025, 2047, 2048, 3071, 3072, 4094, 4095, 4096, 4097, n - 1]:
            if q < n:
                flat[q:] ^= np.uint32(r.integers(1, 1 << 32))
    elif kind in ("cap", "over"):                    # exactly as many change points as a list holds, and one more
        for c0 in range(0, n, CHUNK):
            q = np.sort(r.choice(np.arange(1, min(CHUNK, n - c0)), min(127 + (kind == "over"), n - c0 - 1), replace=False))
            for p in q:
                flat[c0 + p:] ^= np.uint32(1 << int(r.integers(0, 32)))
    elif kind == "short":                            # runs of 1 to 3 in single planes
        q = 0
        while q < n:
            m = int(r.integers(1, 60) if r.random() < 0.6 else r.integers(1, 4))
            flat[q:] ^= np.uint32(int(r.integers(1, 256)) << (8 * int(r.integers(0, 4))))
            q += m
    else:                                            # "noise": every byte differs
        flat[:] = r.integers(0, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32)
    return img


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("w,h", [(4096, 3), (1000, 9), (997, 13), (8193, 1), (3, 1), (130, 70)])
@pytest.mark.parametrize("kind", ["edges", "cap", "over", "short", "noise"])
def test_compressor_paths_match_the_oracle(kind, w, h, mode):
    require_gpu()
    img = _mixed(kind, w, h, [w, h, mode])
    want = oracle.rle_compress(img, mode)
    wide = torch.full((h, w + 3), 77, dtype=torch.int32, device="cuda")
    wide[:, :w] = torch.from_numpy(img.view(np.int32)).cuda()
    for src in (wide[:, :w].contiguous(), wide[:, :w]):              # one run, and rows of another pitch
        buf, size = ec.rle_compress(src.view(torch.uint32), mode)
        ec.default_context().check_status()
        assert buf[:int(size.item())].cpu().numpy().tobytes() == want


@pytest.mark.parametrize("kind", ["noise", "cap"])
@pytest.mark.parametrize("mode", [1, 2])
def test_compressor_with_a_full_pool(kind, mode):
    """The allocation-free entry point's pool holds 512 bytes per chunk of its
    largest image: with every chunk larger, the chunks that find it full are
    coded again when placed."""
    from paper_1902_08755_gb300 import _abi as A
    require_gpu()
    rows = _mixed(kind, 4096, 16, [1, mode])
    img = np.tile(rows, (ec.EC_RLE_CHUNK * 2 // 16, 1)) if kind == "noise" else np.tile(rows, (512, 1))
    img = img[:A.EC_RLE_NOALLOC_MAX_CHUNKS]
    h, w = img.shape
    src = torch.from_numpy(img.view(np.int32)).cuda()
    dst = torch.empty(ec.rle_max_size(w, h), dtype=torch.uint8, device="cuda")
    size, st = torch.zeros(1, dtype=torch.uint64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    A.check(A.load().ec_rle_compress_noalloc(src.data_ptr(), w, h, w, mode, dst.data_ptr(), dst.numel(), size.data_ptr(),
                                             st.data_ptr(), torch.cuda.current_stream().cuda_stream), "noalloc")
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    want = oracle.rle_compress(img, mode)
    assert int(size.item()) == len(want)
    assert dst[:len(want)].cpu().numpy().tobytes() == want
