"""The codec's scratch on a device that is nearly full: where the large pool does
not fit, calls and schedules take the least one and write the same bytes.  The
device is not filled: a preloaded cudaMalloc refuses the sizes it is told to."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_1902_08755_gb300 as ec
from ec_testutil import require_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
size_t refuse_from = (size_t)-1;                 /* sizes from here on do not fit */
int refused;
int cudaMalloc(void** p, size_t n)
{
    static int (*real)(void**, size_t);
    if (n >= refuse_from) { ++refused; return 2; }   /* cudaErrorMemoryAllocation */
    if (!real) real = (int (*)(void**, size_t))dlsym(dlopen("libcudart.so.13", RTLD_NOW), "cudaMalloc");
    return real(p, n);
}
"""

_RUN = r"""
import ctypes as C, sys
import numpy as np, torch
import paper_1902_08755_gb300 as ec
shim = C.CDLL(None)
limit, refused = C.c_size_t.in_dll(shim, "refuse_from"), C.c_int.in_dll(shim, "refused")
img = np.load(sys.argv[1])
src = torch.from_numpy(img.view(np.int32)).cuda().view(torch.uint32)
h, w = img.shape
outs = [(torch.zeros(ec.rle_max_size(w, h), dtype=torch.uint8, device="cuda"),
         torch.zeros(1, dtype=torch.uint64, device="cuda")) for _ in range(6)]
torch.cuda.synchronize()
limit.value = 4 << 20                            # less than a context's first scratch
ctx = ec.Context()
assert refused.value == 1
for i, (dst, size) in enumerate(outs):
    ec.rle_compress(src, i % 3, dst=dst, d_size=size, ctx=ctx)
# a refused size is not asked for again by calls that the scratch is large enough for
assert refused.value == 2, refused.value
limit.value = C.c_size_t(-1).value
ctx.check_status()
for i, (dst, size) in enumerate(outs):
    dst[:int(size.item())].cpu().numpy().tofile(sys.argv[2] + str(i))
ctx.close()

# a schedule's arena
g = torch.Generator(device="cuda")
g.manual_seed(1)
images = []
for k in range(4):
    c = torch.randint(0, 1 << 30, (300, 500), generator=g, device="cuda", dtype=torch.int32)
    d = torch.rand((300, 500), generator=g, device="cuda")
    c[:, 100:400], d[:, 100:400] = k + 1, 0.1 * k
    images.append(ec.Image(c.view(torch.uint32), d))
frames = []
for fits in (True, False):
    oc, od = torch.zeros((300, 500), dtype=torch.int32, device="cuda"), torch.zeros((300, 500), device="cuda")
    torch.cuda.synchronize()
    if not fits:
        limit.value, refused.value = arena, 0
    s = ec.Schedule("depth", "binary_swap", images, oc.view(torch.uint32), od)
    limit.value = C.c_size_t(-1).value
    if fits:
        arena = s.info()["arena_bytes"]
    else:
        assert refused.value == 1 and s.info()["arena_bytes"] < arena
    s.run()
    ec.default_context().check_status()
    frames.append((oc, od, s.stream_sizes()))
    s.close()
assert torch.equal(frames[0][0], frames[1][0]) and torch.equal(frames[0][1], frames[1][1]) and frames[0][2] == frames[1][2]
print("fine")
"""


def test_calls_and_schedules_take_the_least_pool(tmp_path):
    """2048 chunks in turn dense, of few runs and flat: the least pool (512 bytes
    per chunk) has no room for the dense ones, which are coded again when placed."""
    require_gpu()
    r = np.random.default_rng(77)
    img = np.zeros((2048, ec.EC_RLE_CHUNK), np.uint32)
    img[::3] = r.integers(0, 1 << 32, size=img[::3].shape, dtype=np.uint64)
    img[1::3, :100] = r.integers(0, 1 << 32, size=(683, 100), dtype=np.uint64)
    np.save(tmp_path / "img.npy", img)
    (tmp_path / "shim.c").write_text(_SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", tmp_path / "shim.so", tmp_path / "shim.c", "-ldl"], check=True)
    p = subprocess.run([sys.executable, "-c", _RUN, tmp_path / "img.npy", str(tmp_path / "out")], cwd=ROOT,
                       env=dict(os.environ, LD_PRELOAD=str(tmp_path / "shim.so")), capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.strip().endswith("fine"), (p.stdout, p.stderr[-3000:])
    for i in range(6):
        assert (tmp_path / f"out{i}").read_bytes() == oracle.rle_compress(img, i % 3), i
