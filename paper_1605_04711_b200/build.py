"""Builds the CUDA library in-tree, paper_1605_04711_b200/libtwn.so (sm_100a only), and its CPython binding
beside it, _twn.so."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libtwn.so")
BINDING = os.path.join(PKG, "_twn.so")
OBJ = os.path.join(PKG, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.sep not in c or os.path.exists(c)):
            return c
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _torch_dir() -> str:
    import torch
    return os.path.dirname(os.path.abspath(torch.__file__))


def build_binding(force: bool = False) -> str:
    """The host side of the Python calls: csrc/binding.cpp against torch's and CPython's headers."""
    src, hdr = os.path.join(CSRC, "binding.cpp"), os.path.join(ROOT, "include", "twn.h")
    if not force and os.path.exists(BINDING) and os.path.getmtime(BINDING) > max(os.path.getmtime(src), os.path.getmtime(hdr)):
        return BINDING
    inc = os.path.join(_torch_dir(), "include")
    tmp = BINDING + f".{os.getpid()}.tmp"
    subprocess.check_call(["g++", "-O2", "-std=c++20", "-fPIC", "-shared", "-w", "-fvisibility=hidden",
                           "-I", os.path.join(ROOT, "include"), "-I", inc, "-I", os.path.join(inc, "torch", "csrc", "api", "include"),
                           "-I", sysconfig.get_paths()["include"], "-I", "/usr/local/cuda/include", src, "-o", tmp,
                           "-L", PKG, "-l:libtwn.so", "-Wl,-rpath,$ORIGIN", "-L", os.path.join(_torch_dir(), "lib"),
                           "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, BINDING)
    return BINDING


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    deps = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    newest_dep = max(os.path.getmtime(p) for p in deps)
    objs, rebuilt = [], False
    procs = []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), newest_dep):
            cmd = [_nvcc(), *NVCC_FLAGS, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas"); cmd.insert(2, "-v")
            procs.append((src, subprocess.Popen(cmd)))
            rebuilt = True
    for src, p in procs:
        if p.wait() != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    if rebuilt or not os.path.exists(LIB):
        tmp = LIB + f".{os.getpid()}.tmp"
        subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-lcudart", "-ldl"])
        os.replace(tmp, LIB)
    build_binding(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
