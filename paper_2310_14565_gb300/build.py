"""Build the PEPSI CUDA library in-tree: libpepsi_gb300.so next to this file.

nvcc compiles each translation unit for sm_103a only, in parallel, then
links one shared library exporting the C ABI of include/pepsi.h.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJDIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libpepsi_gb300.so")
SOURCES = ["tensor.cu", "relin.cu", "transforms.cu", "client.cu", "mac_planes.cu", "rns.cu", "kernels.cu", "pepsi.cu",
           "engine.cu", "host.cpp"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build the PEPSI library")


def _stale(obj: str, deps) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJDIR, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    headers.append(os.path.join(INCLUDE, "pepsi.h"))
    nv = nvcc()
    common = ["-std=c++17", "-O3", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
    jobs = []
    for src in SOURCES:
        path = os.path.join(CSRC, src)
        obj = os.path.join(OBJDIR, src + ".o")
        if force or _stale(obj, [path] + headers):
            cmd = [nv, "-c", path, "-o", obj] + common
            cmd += ARCH + ["-lineinfo", "--expt-relaxed-constexpr"]
            if not src.endswith(".cu"):
                cmd += ["-x", "cu", "-diag-suppress", "20208"]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("nvcc failed for %s" % cmd[2])

    with cf.ThreadPoolExecutor(max_workers=len(jobs) or 1) as ex:
        list(ex.map(run, jobs))
    objs = [os.path.join(OBJDIR, s + ".o") for s in SOURCES]
    if jobs or force or _stale(LIB, objs):
        tmp = LIB + ".%d.tmp" % os.getpid()
        run([nv, "-shared", "-o", tmp] + objs + ARCH + ["-lcudart"])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
