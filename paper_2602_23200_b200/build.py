"""Builds libinnerq.so (sm_100a) next to this file with nvcc, and the extension module _step (the host side of a step's
calls, against torch's headers; binding.step_path() names its file) with g++.  Usable as `python -m paper_2602_23200_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libinnerq.so")
# every .cu of csrc/: the C ABI, the quantise kernels, the decode kernels (the fused kernel one file per packed format)
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
NVCC_FLAGS = [*ARCH, "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith((".o", ".cpp"))] + [os.path.join(HERE, "..", "include", "innerq.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build_step(force: bool = False) -> str:
    import sysconfig

    import torch

    from .binding import step_path
    src, out, t = os.path.join(CSRC, "innerq_step.cpp"), step_path(), os.path.dirname(torch.__file__)
    if not force and os.path.exists(out) and os.path.getmtime(out) >= max(os.path.getmtime(src), os.path.getmtime(__file__)):
        return out
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I" + sysconfig.get_paths()["include"],
           "-I/usr/local/cuda/include", "-isystem", os.path.join(t, "include"), src, "-o", out,
           "-L" + os.path.join(t, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        _build_lib(verbose)
    try:
        import torch  # noqa: F401
    except ImportError:      # the library alone serves callers of its C ABI
        return LIB
    build_step(force)
    return LIB


def _build_lib(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = list(NVCC_FLAGS)
    if verbose:
        flags += ["-Xptxas", "-v"]
    objs = []
    pending = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        objs.append(obj)
        pending.append([nvcc, *flags, "-c", os.path.join(CSRC, src), "-o", obj])
    # one compiler process per core at a time (there are several dozen translation units: one per packed format)
    jobs = max(1, min(len(pending), os.cpu_count() or 4))
    running = []
    while pending or running:
        while pending and len(running) < jobs:
            cmd = pending.pop(0)
            running.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        cmd, p = running.pop(0)
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            for _, q in running:
                q.kill()
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    cmd = [nvcc, *ARCH, "-shared", "-o", LIB, *objs, "-lcudart"]
    subprocess.run(cmd, check=True)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
