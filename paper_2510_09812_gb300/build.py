"""Build ``libgspm.so`` in-tree for sm_103a (GB300) with nvcc; no CMake, no torch extension.

Translation units compile in parallel; the CUDA runtime is linked statically.
Usage: ``python -m paper_2510_09812_gb300.build`` (or ``build()`` from Python).
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libgspm.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
CUDA_SOURCES = ["cgloop.cu", "kernels.cu", "api.cu", "noalloc.cu", "mpnn.cu"]
CXX_SOURCES = ["host_mesh.cpp"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found (CUDA toolkit required to build libgspm.so)")


def _cuda_home(nvcc: str) -> str:
    return os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))


def _sources():
    return [os.path.join(CSRC, s) for s in CUDA_SOURCES + CXX_SOURCES] + [
        os.path.join(CSRC, "internal.h"), os.path.join(CSRC, "kernels.cuh"),
        os.path.join(CSRC, "device.cuh"),
        os.path.join(CSRC, "flatsum.cuh"), os.path.join(CSRC, "looplayout.h"),
        os.path.join(CSRC, "sum3.h"),
        os.path.join(CSRC, "mpnn.cuh"),
        os.path.join(INCLUDE, "gspm.h")]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(s) <= t for s in _sources())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit and link ``libgspm.so``; returns its path."""
    if not force and up_to_date():
        return LIB
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    common = ["-O3", "-std=c++17", f"-I{INCLUDE}", f"-I{CSRC}"]
    jobs = []
    objs = []
    for s in CUDA_SOURCES:
        o = os.path.join(BUILD, s + ".o")
        objs.append(o)
        jobs.append([nvcc, *ARCH, "-lineinfo", *common,
                     "-Xcompiler", "-fPIC,-fopenmp,-ffp-contract=off",
                     "-Xptxas", "-warn-spills", "-c", os.path.join(CSRC, s), "-o", o])
    for s in CXX_SOURCES:
        o = os.path.join(BUILD, s + ".o")
        objs.append(o)
        # no FMA contraction: the host's dense coarse factorisation and inverse then round alike
        # on x86-64 and aarch64 (GCC contracts a * b + c by default on aarch64 only)
        jobs.append(["g++", *common, f"-I{_cuda_home(nvcc)}/include", "-fPIC", "-fopenmp",
                     "-ffp-contract=off", "-Wall", "-c", os.path.join(CSRC, s), "-o", o])
    procs = [subprocess.Popen(j, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
             for j in jobs]
    failed = []
    for j, p in zip(jobs, procs):
        out, _ = p.communicate()
        if verbose and out:
            sys.stdout.write(out)
        if p.returncode != 0:
            failed.append((j, out))
    if failed:
        msg = "\n".join(" ".join(j) + "\n" + out for j, out in failed)
        raise RuntimeError("libgspm build failed:\n" + msg)
    tmp = LIB + ".tmp"
    link = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-Xcompiler", "-fopenmp", "-lgomp"]
    p = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if p.returncode != 0:
        raise RuntimeError("libgspm link failed:\n" + " ".join(link) + "\n" + p.stdout)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
