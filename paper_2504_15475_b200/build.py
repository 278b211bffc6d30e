"""Compile libersd.so for sm_100a (nvcc cross-compiles without a GPU) and the extension module that
binding.py calls it through, next to this file."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = [os.path.join(HERE, "csrc", "ersd.cu"), os.path.join(HERE, "csrc", "ersd_tree.cpp")]
DEPS = SRC + [os.path.join(HERE, "csrc", "ersd_math.cuh"), os.path.join(HERE, "csrc", "ersd_kernel.inc"), os.path.join(HERE, "csrc", "ersd_cluster.inc"), os.path.join(HERE, "csrc", "ersd_cluster_top.inc"), os.path.join(HERE, "csrc", "ersd_gsd.inc"), os.path.join(ROOT, "include", "ersd.h")]
LIB = os.path.join(HERE, "libersd.so")
CALL_SRC = os.path.join(HERE, "csrc", "ersd_call.cpp")
CALL_LIB = os.path.join(HERE, "_ersd_call.so")  # the calling side of binding.py


def nvcc_command(out: str, extra=()):
    # (--no-compress: unpacking the device code was half of the 28 ms that a process's first launch took; 13 without it)
    return ["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "--no-compress", "-std=c++17",
            "--shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
            "-I", os.path.join(HERE, "csrc"), *extra, "-o", out, *SRC]


def call_command(out: str):
    """g++ line of the extension module behind binding.py (built against the installed torch)."""
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    return ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            '-DERSD_TORCH_VERSION="%s"' % torch.__version__,
            "-I", os.path.join(ROOT, "include"), "-I", os.path.join(root, "include"),
            "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
            "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), CALL_SRC, "-o", out,
            "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _fresh(lib: str, deps) -> bool:
    return os.path.exists(lib) and all(os.path.getmtime(lib) >= os.path.getmtime(d) for d in deps)


def _call_fresh() -> bool:
    """Whether the extension module is newer than its sources and built against the installed torch."""
    import torch
    if not _fresh(CALL_LIB, [CALL_SRC, os.path.join(ROOT, "include", "ersd.h")]):
        return False
    with open(CALL_LIB, "rb") as f:
        return b"\0" + str(torch.__version__).encode() + b"\0" in f.read()


def build(force: bool = False, verbose: bool = False) -> str:
    jobs = []
    if force or not _fresh(LIB, DEPS):
        jobs.append((LIB, lambda out: nvcc_command(out, ("-Xptxas", "-v") if verbose else ())))
    if force or not _call_fresh():
        jobs.append((CALL_LIB, call_command))
    running = []
    for lib, command in jobs:
        tmp = lib + ".tmp.%d" % os.getpid()
        running.append((lib, tmp, subprocess.Popen(command(tmp))))
    for lib, tmp, job in running:
        if job.wait() != 0:
            raise RuntimeError("building %s failed" % lib)
        os.replace(tmp, lib)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
