"""Compile the CUDA sources under csrc/ into libaccerl.so (in-tree) with nvcc for sm_100a, and the
Python module of the hot calls (csrc/torch_calls.cpp) against it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
SO = os.path.join(HERE, "libaccerl.so")
CALLS = os.path.join(HERE, "_calls.so")

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC,-ffp-contract=off,-fno-fast-math,-falign-functions=64,-falign-loops=32", "-cudart", "static",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _build_calls(force: bool) -> str:
    """The Python module of the hot calls: one C++ file against torch's headers and libaccerl.so."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    src = os.path.join(CSRC, "torch_calls.cpp")
    if force or _stale(CALLS, [src, os.path.join(ROOT, "include", "accerl.h")]):
        lib = os.path.join(os.path.dirname(torch.__file__), "lib")
        inc = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], *cpp_extension.include_paths("cuda")]
        tmp = CALLS + ".%d.tmp" % os.getpid()
        subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", tmp,
                               "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
                               *["-isystem" + i for i in inc], "-L" + HERE, "-laccerl", "-L" + lib, "-ltorch_python",
                               "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda",
                               "-Wl,-rpath,$ORIGIN"])
        os.replace(tmp, CALLS)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    """Build (if stale) and return the path of libaccerl.so."""
    os.makedirs(OBJ, exist_ok=True)
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = (glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) +
               glob.glob(os.path.join(ROOT, "include", "*.h")))
    objs, cmds = [], []
    for src in sources:
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            cmd = [NVCC, *FLAGS, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
                print(" ".join(cmd), file=sys.stderr)
            cmds.append(cmd)
    with ThreadPoolExecutor(os.cpu_count() or 1) as pool:
        list(pool.map(subprocess.check_call, cmds))
    if force or _stale(SO, objs):
        tmp = SO + ".%d.tmp" % os.getpid()
        # (nodelete: a thread of the library may be asleep in it when a program closes it)
        subprocess.check_call([NVCC, "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                               "-Xlinker", "-z", "-Xlinker", "nodelete", "-o", tmp, *objs])
        os.replace(tmp, SO)
    _build_calls(force)
    return SO


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
