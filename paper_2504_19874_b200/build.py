"""Builds libtq.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _tqbind.so (the marshalling half of the
Python binding) with the host compiler."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
LIB = os.path.join(PKG, "libtq.so")
LIB_DEBUG = os.path.join(PKG, "libtq_debug.so")   # the same sources with -DTQ_DEBUG (device-side index checks)


BIND = os.path.join(PKG, "_tqbind.so")
BIND_SRC = os.path.join(PKG, "csrc", "tq_bind.cpp")


def sources():
    return sorted(glob.glob(os.path.join(PKG, "csrc", "*.cu")))


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(PKG, "csrc", "*.h")) + glob.glob(os.path.join(PKG, "csrc", "*.cuh"))
    deps += glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return any(os.path.getmtime(p) > t for p in deps)


def build_binding(force: bool = False) -> str:
    header = os.path.join(ROOT, "include", "tq.h")
    if not force and os.path.exists(BIND) and all(os.path.getmtime(p) <= os.path.getmtime(BIND) for p in (BIND_SRC, header)):
        return BIND
    import torch
    torch_dir = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(torch_dir, "include"),
           "-isystem", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
           "-I", sysconfig.get_paths()["include"], BIND_SRC, "-o", BIND, "-L", os.path.join(torch_dir, "lib"),
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-L", os.path.join(cuda, "lib64"), "-lcudart", "-ldl"]
    subprocess.run(cmd, check=True)
    return BIND


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib = LIB_DEBUG if debug else LIB
    build_binding(force)
    if not force and not _stale(lib):
        return lib
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    bdir = os.path.join(PKG, "_build_debug" if debug else "_build")
    os.makedirs(bdir, exist_ok=True)
    for src in sources():
        obj = os.path.join(bdir, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
               "-Xcompiler", "-fPIC,-fopenmp,-Wall", "-I", os.path.join(ROOT, "include"),
               "-I", os.path.join(PKG, "csrc"), "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        if debug:
            cmd.insert(1, "-DTQ_DEBUG")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip() and (verbose or p.returncode != 0):
            sys.stderr.write(out)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    link = [nvcc, "-shared", "-o", lib] + objs + ["-lgomp", "-ldl"]
    subprocess.run(link, check=True)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
