"""Build the CUDA library in-tree with nvcc for sm_100a, and the small module that calls it on torch tensors.

``python -m paper_2211_10526_b200.build`` (or ``build()``) compiles every ``.cu`` file under
``csrc/`` into ``libcastling_attn.so`` beside this module, and ``csrc/torch_call.cpp`` into
``_torch_call.so``.  nvcc cross-compiles, so no GPU is needed to build.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB_PATH = os.path.join(_HERE, "libcastling_attn.so")
CALL_SOURCE = os.path.join(CSRC, "torch_call.cpp")
CALL_PATH = os.path.join(_HERE, "_torch_call.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def _start_torch_call(verbose: bool) -> subprocess.Popen:
    """g++ on the torch-facing module; its symbols of torch resolve against the libraries torch has loaded."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DBUILT_AGAINST="{_torch_tag().decode()}"', "-I", INCLUDE,
           "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], CALL_SOURCE, "-o",
           f"{CALL_PATH}.{os.getpid()}.tmp", "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    if verbose:
        print(" ".join(cmd), file=sys.stderr)
    return subprocess.Popen(cmd)


def _torch_tag() -> bytes:
    import torch
    return f"built against torch {torch.__version__}".encode()


def _call_stale() -> bool:
    if not os.path.exists(CALL_PATH):
        return True
    with open(CALL_PATH, "rb") as f:   # another torch may have another C++ interface
        if _torch_tag() + b"\0" not in f.read():
            return True
    built = os.path.getmtime(CALL_PATH)
    return any(os.path.getmtime(p) > built for p in [CALL_SOURCE] + glob.glob(os.path.join(INCLUDE, "*.h")))


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Compile what is stale and return the path of the shared library."""
    call = _start_torch_call(verbose) if force or _call_stale() else None
    try:
        return _build_library(force, verbose, extra_flags)
    finally:
        if call is not None:
            if call.wait() != 0:
                raise RuntimeError(f"the C++ compiler failed on {CALL_SOURCE}")
            os.replace(f"{CALL_PATH}.{os.getpid()}.tmp", CALL_PATH)


def _build_library(force: bool, verbose: bool, extra_flags) -> str:
    if not force and not _stale():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    for src in sources():
        obj = os.path.join(CSRC, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc, *NVCC_FLAGS, *extra_flags, "-I", INCLUDE, "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        procs.append((src, subprocess.Popen(cmd)))
        objs.append(obj)
    for src, proc in procs:
        if proc.wait() != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = f"{LIB_PATH}.{os.getpid()}.tmp"
    cmd = [nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a", "-lcudart_static"]
    if verbose:
        print(" ".join(cmd), file=sys.stderr)
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
