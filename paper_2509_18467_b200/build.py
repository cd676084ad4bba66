"""Builds ``liblawcat.so`` (the C-ABI CUDA library, nvcc for sm_100a) and ``_binding.so`` (the CPython module in front of it,
g++) in-tree.

Usage: ``python -m paper_2509_18467_b200.build [--force] [--verbose]``.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "liblawcat.so")
BINDING = os.path.join(PKG, "_binding.so")  # the CPython module that marshals tensors (csrc/binding.cpp)
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

# (no fast-math: the exact path relies on the precise division, exp and log of the default settings)
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _newest_header():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(ROOT, "include", "lawcat.h"))
    return max(os.path.getmtime(h) for h in hs)


def _binding_cmd():
    import sysconfig

    from torch.utils import cpp_extension
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    libs = cpp_extension.library_paths()
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", os.path.join(CSRC, "binding.cpp"), "-o", BINDING,
            *[f"-I{d}" for d in inc], *[f"-L{d}" for d in libs], *[f"-Wl,-rpath,{d}" for d in libs],
            "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    hdr = _newest_header()
    jobs = []
    binding = os.path.join(CSRC, "binding.cpp")
    build_binding = force or not os.path.exists(BINDING) or os.path.getmtime(BINDING) < os.path.getmtime(binding)
    for s in sources():
        src, obj = os.path.join(CSRC, s), os.path.join(OBJ, s[:-3] + ".o")
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr):
            cmd = [NVCC, *FLAGS, "-Xptxas", "-v", "-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("compiler failed: " + " ".join(cmd))
        if "-c" in cmd:  # registers, spills and shared memory of every kernel, beside the object
            with open(cmd[-1][:-2] + ".ptxas", "w") as f:
                f.write(r.stderr)

    with ThreadPoolExecutor(max_workers=8) as ex:
        list(ex.map(run, jobs + ([_binding_cmd()] if build_binding else [])))
    objs = [os.path.join(OBJ, s[:-3] + ".o") for s in sources()]
    if jobs or not os.path.exists(LIB):
        run([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs])
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
