"""Builds libmoe_b200.so in-tree with nvcc for sm_100a (no JIT cache), and _fastcall, the step calls' way in from Python."""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

from .binding import fastcall_path

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
OUT = os.path.join(PKG, "libmoe_b200.so")
OBJ = os.path.join(PKG, "_build")
SOURCES = ["api.cu", "route_layout.cu", "permute.cu", "gemm_tc3.cu", "gemm_wgrad.cu", "fused.cu", "study.cu", "router.cu", "taskflow.cu", "ep.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        path = cand and shutil.which(cand)
        if path:
            return path
    raise RuntimeError("nvcc not found")


def _cuda_include() -> str:
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")


def _stale(out: str) -> bool:
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    inc = os.path.join(PKG, "..", "include")
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(inc, f) for f in os.listdir(inc)]
    return any(os.path.getmtime(d) > t for d in deps)


def _compile(src: str) -> str:
    obj = os.path.join(OBJ, src.replace(".cu", ".o"))
    cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    with open(obj + ".log", "w") as f:
        f.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}{r.stderr}")
    return obj


def _build_fastcall() -> None:
    import torch
    root, path = os.path.dirname(torch.__file__), fastcall_path()
    tmp = path + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-I" + sysconfig.get_paths()["include"], "-I" + _cuda_include(),
           os.path.join(CSRC, "fastcall.cpp"), "-o", tmp, "-L" + os.path.join(root, "lib"),
           "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on fastcall.cpp:\n{r.stdout}{r.stderr}")
    os.replace(tmp, path)


def _try_fastcall() -> None:
    """The library does not need it (the binding then checks its arguments in Python), so a box without a C++ compiler, Python's
    or torch's headers goes without; what an older source left there is not kept."""
    try:
        _build_fastcall()
    except (OSError, RuntimeError, ImportError) as e:
        if os.path.exists(fastcall_path()):
            os.unlink(fastcall_path())
        warnings.warn(f"calls from Python go the slower way, the accelerator could not be built: {e}")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source for sm_100a and link the C-ABI shared library.  Returns its path."""
    lib, fast = force or _stale(OUT), force or _stale(fastcall_path())
    if not (lib or fast):
        return OUT
    os.makedirs(OBJ, exist_ok=True)
    with concurrent.futures.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
        side = ex.submit(_try_fastcall) if fast else None
        objs = list(ex.map(_compile, SOURCES)) if lib else []
        if side:
            side.result()
    if lib:
        tmp = OUT + f".tmp{os.getpid()}"
        cmd = [_nvcc(), "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
        subprocess.check_call(cmd)
        os.replace(tmp, OUT)
    if verbose:
        for o in objs:
            sys.stdout.write(open(o + ".log").read())
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
