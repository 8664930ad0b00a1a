"""Builds ``libtaq.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

``python -m paper_2603_22943_b200.build`` or ``build_library()``.  Objects go to ``_build/`` inside the package;
a source is recompiled only when it (or a header) is newer than its object.  ``_taq_call.so``, the binding's native call
path, is built beside it.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libtaq.so")
CALL_SRC = os.path.join(CSRC, "taq_pymodule.cpp")
CALL = os.path.join(PKG, "_taq_call.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v", "--expt-relaxed-constexpr",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found; the TAQ library needs the CUDA toolkit to build")
    return exe


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _newest_header() -> float:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(ROOT, "include", "taq.h"))
    return max(os.path.getmtime(h) for h in hs)


def build_library(force: bool = False, verbose: bool = False, profile: bool = False) -> str:
    """``profile=True`` builds ``libtaq_profile.so`` with the phase stamps of ``csrc/taq_prof.cuh`` compiled in
    (into its own object directory); the normal library contains none of that code."""
    if profile:
        return _build(os.path.join(PKG, "_build_profile"), os.path.join(PKG, "libtaq_profile.so"), ["-DTAQ_PROFILE"], True, verbose)
    build_call_module(force)
    return _build(BUILD, LIB, [], force, verbose)


def build_call_module(force: bool = False) -> str:
    """Compiles ``_taq_call.so``, the binding's native call path (CPython and torch headers, host compiler only)."""
    import sysconfig
    import torch
    newest = max(os.path.getmtime(CALL_SRC), os.path.getmtime(os.path.join(ROOT, "include", "taq.h")))
    if not force and os.path.exists(CALL) and os.path.getmtime(CALL) >= newest:
        return CALL
    troot = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(troot, "include"), "-I", os.path.join(troot, "include", "torch", "csrc", "api", "include"),
           "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], CALL_SRC, "-o", CALL,
           "-L", os.path.join(troot, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    if p.returncode != 0:
        raise RuntimeError(f"g++ failed on {CALL_SRC}:\n{p.stdout}\n{p.stderr}")
    return CALL


def _build(BUILD: str, LIB: str, extra: list, force: bool, verbose: bool) -> str:
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    hdr_time = _newest_header()
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time):
            jobs.append((src, obj))

    def compile_one(job):
        src, obj = job
        cmd = [nvcc] + NVCC_FLAGS + extra + ["-c", src, "-o", obj]
        p = subprocess.run(cmd, capture_output=True, text=True)
        log = os.path.join(BUILD, os.path.basename(src)[:-3] + ".log")
        with open(log, "w") as f:
            f.write(" ".join(cmd) + "\n" + p.stdout + p.stderr)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{p.stdout}\n{p.stderr}")
        if verbose:
            sys.stderr.write(p.stderr)
        return obj

    if jobs:
        with ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            list(ex.map(compile_one, jobs))
    if jobs or not os.path.exists(LIB):
        cmd = [nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        p = subprocess.run(cmd, capture_output=True, text=True)
        if p.returncode != 0:
            raise RuntimeError(f"link failed:\n{p.stdout}\n{p.stderr}")
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose=True, profile="--profile" in sys.argv))
