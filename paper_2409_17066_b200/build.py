"""Build libvptq.so (sm_100a only) with nvcc and the extension module _native with g++, both in-tree."""
from __future__ import annotations

import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libvptq.so")
NATIVE = os.path.join(HERE, "_native.so")          # CPython extension: tensors -> the C ABI
NATIVE_SRC = os.path.join(CSRC, "native_binding.cpp")
OBJ = os.path.join(HERE, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        [os.path.join(os.path.dirname(HERE), "include", "vptq.h")]


def build_native(force: bool = False) -> str:
    """Compile the extension module against torch's headers; it links libvptq.so next to it."""
    deps = [NATIVE_SRC, os.path.join(os.path.dirname(HERE), "include", "vptq.h")]
    if not force and os.path.exists(NATIVE) and os.path.getmtime(NATIVE) >= max(os.path.getmtime(p) for p in deps):
        return NATIVE
    import sysconfig
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [sysconfig.get_paths()["include"], os.path.join(root, "include"),
           os.path.join(root, "include", "torch", "csrc", "api", "include"), "/usr/local/cuda/include"]
    cmd = ["g++", "-O2", "-std=c++20", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *[f"-I{i}" for i in inc], NATIVE_SRC, "-o", NATIVE, f"-L{HERE}", f"-L{os.path.join(root, 'lib')}", "-l:libvptq.so",
           "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10", "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/, link libvptq.so next to this file, and build the extension module."""
    lib = build_library(force, verbose)
    build_native(force)
    return lib


def build_library(force: bool = False, verbose: bool = False) -> str:
    newest = max(os.path.getmtime(p) for p in _deps())
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    os.makedirs(OBJ, exist_ok=True)
    hdr_time = max(os.path.getmtime(p) for p in _deps() if not p.endswith(".cu"))
    objs, procs = [], []
    for src in _sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if (not force and os.path.exists(obj)
                and os.path.getmtime(obj) >= max(os.path.getmtime(src), hdr_time)):
            continue
        cmd = ["nvcc"] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = []
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            print(out)
        if pr.returncode != 0:
            failed.append(src)
    if failed:
        raise RuntimeError("nvcc failed for: " + ", ".join(failed))
    subprocess.run(["nvcc", "-shared", "-gencode", "arch=compute_100a,code=sm_100a",
                    "-o", LIB] + objs, check=True)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
