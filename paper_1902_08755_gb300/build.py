"""Build libec.so (the CUDA library behind include/ec.h) in-tree with nvcc, and
the binding's argument marshalling (_marshal.*.so) with the host compiler.

Every translation unit is compiled for sm_103a only, in parallel, then linked
into paper_1902_08755_gb300/libec.so.  No cmake; either library is rebuilt when
one of its sources is newer.  The marshalling module reads torch's and Python's
own object layouts, so its file name carries both versions and it is built again
for others.  The library does not need it: without a host compiler or Python's
headers the build warns, and the binding checks its arguments in Python.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig
import warnings
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libec.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2", "--expt-relaxed-constexpr",
         "-I", os.path.join(ROOT, "include")]


def _nvcc() -> str:
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    p = os.path.join(home, "bin", "nvcc")
    return p if os.path.exists(p) else "nvcc"


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def marshal_path() -> str:
    """The marshalling module of this interpreter and this torch."""
    import torch
    return os.path.join(HERE, f"_marshal.torch-{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def _older(path, deps) -> bool:
    return not os.path.exists(path) or any(os.path.exists(p) and os.path.getmtime(p) > os.path.getmtime(path) for p in deps)


def _headers():
    return glob.glob(os.path.join(ROOT, "include", "*.h"))


def _stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def marshal_stale() -> bool:
    return _older(marshal_path(), [os.path.join(CSRC, "marshal.cpp")] + _headers())


def _build_marshal() -> None:
    import torch
    troot = os.path.dirname(torch.__file__)
    tmp = marshal_path() + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(troot, "include"),
           os.path.join(CSRC, "marshal.cpp"), "-o", tmp,
           "-L", os.path.join(troot, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for marshal.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, marshal_path())


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    lib, marshal = force or _stale(), force or marshal_stale()
    with ThreadPoolExecutor(max_workers=min(12, os.cpu_count() or 1)) as ex:
        m = ex.submit(_build_marshal) if marshal else None
        if lib:
            _build_lib(ex, verbose, extra)
        try:
            if m is not None:
                m.result()
        except (OSError, RuntimeError) as e:
            warnings.warn(f"the native argument marshalling was not built (arguments are checked in Python): {e}")
    return LIB


def _build_lib(ex, verbose, extra) -> None:
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src).replace(".cu", ".o"))
        cmd = [nvcc, *ARCH, *FLAGS, *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr)
        return obj

    objs = list(ex.map(compile_one, sources()))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True,
                extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else []))
