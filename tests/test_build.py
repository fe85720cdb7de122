"""Building and loading: the CUDA library and the binding's marshalling module
depend on their own sources and tools only, and the binding works without the
module."""
import os
import subprocess
import sysconfig

import pytest
import torch

from paper_1902_08755_gb300 import _abi as A
from paper_1902_08755_gb300 import api
from paper_1902_08755_gb300 import build as B


@pytest.fixture
def tools(monkeypatch, tmp_path):
    """Compilers that write empty files into tmp_path; `fails` names the ones that fail."""
    fails, ran = set(), []

    def run(cmd, **kw):
        tool = os.path.basename(cmd[0])
        ran.append(tool)
        if tool in fails:
            return subprocess.CompletedProcess(cmd, 1, "", "no such header")
        if tool + " missing" in fails:
            raise FileNotFoundError(tool)
        open(cmd[cmd.index("-o") + 1], "w").close()
        return subprocess.CompletedProcess(cmd, 0, "", "")
    monkeypatch.setattr(B.subprocess, "run", run)
    monkeypatch.setattr(B, "LIB", str(tmp_path / "libec.so"))
    monkeypatch.setattr(B, "BUILD", str(tmp_path / "_build"))
    monkeypatch.setattr(B, "HERE", str(tmp_path))
    return fails, ran


@pytest.mark.parametrize("fail", ["g++", "g++ missing"])
def test_the_library_does_not_need_the_host_compiler(tools, fail):
    fails, ran = tools
    fails.add(fail)
    with pytest.warns(UserWarning, match="not built"):
        B.build()
    assert os.path.exists(B.LIB) and not os.path.exists(B.marshal_path())
    # the library is not compiled again for the module's sake
    n = ran.count("nvcc")
    fails.clear()
    B.build()
    assert os.path.exists(B.marshal_path()) and ran.count("nvcc") == n
    ran.clear()
    B.build()
    assert not ran


def test_the_module_does_not_need_the_cuda_compiler(tools):
    fails, ran = tools
    fails.add("nvcc")
    with pytest.raises(RuntimeError, match="nvcc failed"):
        B.build()
    assert os.path.exists(B.marshal_path())


def test_the_module_belongs_to_its_python_and_torch(tools, monkeypatch):
    B.build()
    path = B.marshal_path()
    assert path.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and torch.__version__ in os.path.basename(path)
    assert not B.marshal_stale()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert B.marshal_stale() and not B._stale()


def test_older_module_is_stale(tools):
    B.build()
    os.utime(B.marshal_path(), (1, 1))
    assert B.marshal_stale() and not B._stale()
    os.utime(B.LIB, (1, 1))
    assert B._stale()


@pytest.mark.parametrize("how", ["missing", "unloadable"])
def test_arguments_are_checked_in_python_without_the_module(monkeypatch, tmp_path, how):
    path = tmp_path / "_marshal.so"
    if how == "unloadable":
        path.write_bytes(b"built for another machine")
    monkeypatch.setattr(A, "_marshal", None)
    monkeypatch.setattr(A, "load", lambda: None)
    monkeypatch.setattr(B, "marshal_path", lambda: str(path))
    monkeypatch.setattr(api, "_on_device", lambda *a: None)
    color, depth = torch.zeros((4, 6), dtype=torch.int32), torch.ones((4, 6))
    with pytest.warns(UserWarning, match="not used"):
        arr = api._images([api.Image(color, depth, (1, 2, 6, 4))], 0, api._DEPTH)
    assert (arr[0].pvp.x, arr[0].pvp.h, arr[0].color, arr[0].depth) == (1, 4, color.data_ptr(), depth.data_ptr())
    assert api._target(color, depth, None, 0).color == color.data_ptr()
    assert list(api._order([1, 0], 2)) == [1, 0]
    g = torch.zeros((4, 6, 4))
    assert list(api._gradients([g], [api.Image(torch.zeros((4, 6, 4)))], 0)[1]) == [g.data_ptr()]
