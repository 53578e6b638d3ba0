"""The build: the library comes out without the accelerator of the Python calls."""
import ctypes
import os
import re
import shutil

import pytest
import torch

from paper_2605_23764_b200 import binding, build


def test_library_is_built_without_the_accelerator(monkeypatch, tmp_path):
    build.build()
    compiled = build.OBJ

    def no_compiler():
        raise FileNotFoundError("g++")

    def compile_(src):   # the objects are there
        obj = src.replace(".cu", ".o")
        return shutil.copy(os.path.join(compiled, obj), tmp_path / obj)
    monkeypatch.setattr(build, "OBJ", str(tmp_path))
    monkeypatch.setattr(build, "OUT", str(tmp_path / "lib.so"))
    monkeypatch.setattr(build, "fastcall_path", lambda: str(tmp_path / "fast.so"))
    monkeypatch.setattr(build, "_compile", compile_)
    monkeypatch.setattr(build, "_build_fastcall", no_compiler)
    (tmp_path / "fast.so").write_bytes(b"of an older source")
    with pytest.warns(UserWarning, match="g\\+\\+"):
        out = build.build(force=True)
    assert hasattr(ctypes.CDLL(out), "moe_create")
    assert not (tmp_path / "fast.so").exists()


def test_cuda_headers_are_found_from_a_bare_nvcc(monkeypatch):
    nvcc = build._nvcc()
    monkeypatch.setenv("NVCC", "nvcc")
    monkeypatch.setenv("PATH", os.path.dirname(nvcc) + os.pathsep + os.environ.get("PATH", ""))
    assert os.path.isabs(build._nvcc())
    assert os.path.exists(os.path.join(build._cuda_include(), "cuda_runtime.h"))


def test_accelerator_of_another_torch_or_python_is_not_taken(monkeypatch):
    build.build()
    path = build.fastcall_path()
    assert os.path.exists(path) and not build._stale(path)
    assert binding._load_fastcall() is not None
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0.1")
        assert build._stale(build.fastcall_path()) and binding._load_fastcall() is None
    with monkeypatch.context() as m:
        m.setattr(binding.sysconfig, "get_config_var", lambda name: ".cpython-399-other.so")
        assert build._stale(build.fastcall_path()) and binding._load_fastcall() is None


def test_persistent_kernels_hardly_spill():
    """The backward's epilogue takes every register of the 128 a thread has: what a role carries besides it spills, and 32 bytes of
    that made a backward over a thousand tokens 4 % slower.  At most 16 bytes; the forward none."""
    build.build()
    with open(os.path.join(build.OBJ, "fused.o.log")) as f:
        log = f.read()
    spills = {m[0]: int(m[1]) for m in re.findall(r"fused_chain_kernelILb(\d)E.*?\n.*?(\d+) bytes spill stores", log)}
    assert spills["0"] == 0 and spills["1"] <= 16, spills
