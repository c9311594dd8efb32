"""Builds the CUDA library (libpc.so, sm_100a only) and the native call wrappers (_pc_calls.so) in-tree."""
from __future__ import annotations

import importlib.metadata
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpc.so")
SOURCES = ["pc_api.cu"]
CALLS = os.path.join(HERE, "_pc_calls.so")
CALLS_SOURCE = os.path.join(CSRC, "py_calls.cpp")


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [os.path.join(HERE, "..", "include", "pc.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def calls_key() -> str:
    """What the call wrappers are compiled against beside their source: torch's C++ ABI and this interpreter's.  The text is
    compiled in (the module's built_for)."""
    return f"built for torch {importlib.metadata.version('torch')}, python {sys.version_info.major}.{sys.version_info.minor}"


def _calls_stale() -> bool:
    if not os.path.exists(CALLS):
        return True
    t = os.path.getmtime(CALLS)
    if any(os.path.getmtime(d) > t for d in (CALLS_SOURCE, os.path.join(HERE, "..", "include", "pc.h"), __file__)):
        return True
    with open(CALLS, "rb") as f:
        return calls_key().encode() + b"\0" not in f.read()


def build_calls(force: bool = False) -> str:
    """The CPython extension of csrc/py_calls.cpp (host code only)."""
    if not force and not _calls_stale():
        return CALLS
    import torch
    from torch.utils import cpp_extension
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DPC_CALLS_KEY="{calls_key()}"']
    for inc in cpp_extension.include_paths() + [sysconfig.get_paths()["include"], cuda]:
        cmd += ["-isystem", inc]
    cmd += [CALLS_SOURCE, "-o", CALLS, "-L" + lib, "-ltorch_python", "-lc10", "-lc10_cuda", "-Wl,-rpath," + lib]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    build_calls(force)
    if not force and not _stale():
        return LIB
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "-cudart", "static",
           "-DPC_BUILDING_LIB"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
