"""Builds the CUDA library (``libhikonv.so``) for sm_100a with nvcc, in-tree.

Every translation unit under ``csrc/`` is compiled to an object under ``_build/`` (only when it or a header is
newer than the object), side by side, and the objects are linked into one shared library.  The fast path of the Python
binding (``pyext/fast.cpp``) is a second library, an extension module that uses PyTorch's tensors; it is compiled beside them.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ_DIR = os.path.join(HERE, "_build")
LIB_PATH = os.path.join(HERE, "libhikonv.so")
EXT_SRC = os.path.join(HERE, "pyext", "fast.cpp")
EXT_PATH = os.path.join(HERE, "_fast" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17", "--use_fast_math",
    "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cpp")))


def _headers():
    return (glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh"))
            + glob.glob(os.path.join(ROOT, "include", "*.h")))


def _object_of(src: str) -> str:
    return os.path.join(OBJ_DIR, os.path.basename(src) + ".o")


def _build_extension(force: bool, verbose: bool) -> None:
    """The extension module of the binding (host code only)."""
    deps = [EXT_SRC] + glob.glob(os.path.join(ROOT, "include", "*.h"))
    if not force and os.path.exists(EXT_PATH) and os.path.getmtime(EXT_PATH) >= max(os.path.getmtime(d) for d in deps):
        return
    import torch
    from torch.utils import cpp_extension
    torch_lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    includes = cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
    tmp = EXT_PATH + ".tmp.%d" % os.getpid()
    cmd = ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", EXT_SRC, "-o", tmp,
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
           + ["-I" + i for i in includes] + ["-L" + torch_lib, "-Wl,-rpath," + torch_lib]
           + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    if verbose:
        print(" ".join(cmd), flush=True)
    subprocess.run(cmd, check=True)
    os.replace(tmp, EXT_PATH)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Compile what is out of date under csrc/ and link the shared library; a no-op when nothing changed."""
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    newest_header = max(os.path.getmtime(h) for h in _headers())
    flags = NVCC_FLAGS + list(extra_flags) + ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    stale = [s for s in sources()
             if force or extra_flags or not os.path.exists(_object_of(s))
             or os.path.getmtime(_object_of(s)) < max(os.path.getmtime(s), newest_header)]

    def compile_one(src: str) -> None:
        cmd = [nvcc] + flags + ["-c", src, "-o", _object_of(src)]
        if verbose:
            print(" ".join(cmd), flush=True)
        subprocess.run(cmd, check=True)

    # the longest compilations first
    stale.sort(key=lambda s: ("strip" not in s, "small" not in s))
    with ThreadPoolExecutor(max_workers=max(2, min(len(stale) + 1, os.cpu_count() or 4))) as pool:
        ext = pool.submit(_build_extension, force, verbose)
        list(pool.map(compile_one, stale))
        ext.result()
    objects = [_object_of(s) for s in sources()]
    if stale or not os.path.exists(LIB_PATH) or os.path.getmtime(LIB_PATH) < max(os.path.getmtime(o) for o in objects):
        tmp = LIB_PATH + ".tmp.%d" % os.getpid()
        cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objects
        if verbose:
            print(" ".join(cmd), flush=True)
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    flags = ["-Xptxas", "-v"] if "--ptxas" in sys.argv else []
    print(build(force="--force" in sys.argv, verbose=True, extra_flags=flags))
