"""Compile libersd.so for sm_100a (nvcc cross-compiles without a GPU) and the extension module that
binding.py calls it through, next to this file."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
SRC = [os.path.join(CSRC, name) for name in ("ersd.cu", "ersd_cluster_bf16.cu", "ersd_cluster_f32.cu", "ersd_tree.cpp")]
DEPS = SRC + [os.path.join(CSRC, name) for name in ("ersd_device.cuh", "ersd_math.cuh", "ersd_kernel.inc", "ersd_cluster.inc",
                                                    "ersd_cluster_top.inc", "ersd_cluster_select.inc", "ersd_gsd.inc")]
DEPS.append(os.path.join(ROOT, "include", "ersd.h"))
LIB = os.path.join(HERE, "libersd.so")
CALL_SRC = os.path.join(HERE, "csrc", "ersd_call.cpp")
CALL_LIB = os.path.join(HERE, "_ersd_call.so")  # the calling side of binding.py


def nvcc_command(out: str, inputs, extra=()):
    # (--no-compress: unpacking the device code was half of the 28 ms that a process's first launch took; 13 without it)
    return ["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "--no-compress", "-std=c++17",
            "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC, *extra, "-o", out, *inputs]


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


def _wait(jobs) -> None:
    failed = [what for what, job in jobs if job.wait() != 0]  # (all have ended by then)
    if failed:
        raise RuntimeError("building %s failed" % ", ".join(failed))


def build(force: bool = False, verbose: bool = False) -> str:
    tag = ".tmp.%d" % os.getpid()
    running, objects = [], []
    new_lib, new_call = force or not _fresh(LIB, DEPS), force or not _call_fresh()
    if new_lib:
        for src in SRC:
            objects.append(os.path.join(HERE, os.path.basename(src) + tag + ".o"))
            running.append((src, subprocess.Popen(nvcc_command(objects[-1], ["-c", src], ("-Xptxas", "-v") if verbose else ()))))
    if new_call:
        running.append((CALL_LIB, subprocess.Popen(call_command(CALL_LIB + tag))))
    try:
        _wait(running)
        if new_lib:
            _wait([(LIB, subprocess.Popen(nvcc_command(LIB + tag, ["--shared", *objects])))])
            os.replace(LIB + tag, LIB)
        if new_call:
            os.replace(CALL_LIB + tag, CALL_LIB)
    finally:
        for path in objects:
            if os.path.exists(path):
                os.remove(path)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
