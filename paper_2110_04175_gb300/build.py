"""Builds librelaysum.so in-tree with nvcc for sm_103a (GB300).

Translation units compiled in parallel (host program builder, C ABI with the
setup kernels, host-state step, and the step kernels once per capacity),
linked into one shared library with the CUDA runtime statically linked, so the
library loads on a machine without a GPU.
"""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "librelaysum.so")

# (source, its own flags): the step kernels are built for up to 64 workers
# (relaysum::kSmallN) and for up to 256 (relaysum::kMaxN)
SOURCES = [("step_kernels.cu", ["-DRELAY_CAP=256", "-DRELAY_SPACE=large"]),
           ("step_kernels.cu", ["-DRELAY_CAP=64", "-DRELAY_SPACE=small"]),
           ("relaysum.cu", []), ("program.cpp", []), ("host_step.cpp", [])]
HEADERS = [os.path.join(CSRC, h) for h in ("program.h", "handle.h", "device.cuh", "step_launch.h")] + [
    os.path.join(INCLUDE, "relaysum.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
              "-I" + INCLUDE, "-I" + CSRC]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build librelaysum.so")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s, _ in SOURCES] + HEADERS + [os.path.abspath(__file__)]
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles (if stale) and returns the path of librelaysum.so."""
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    tag = str(os.getpid())

    def compile_one(unit) -> str:
        src, flags = unit
        obj = os.path.join(BUILD, f"{src}{''.join(flags[:1])}.{tag}.o")
        cmd = [cc, *ARCH, *NVCC_FLAGS, *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    with concurrent.futures.ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".{tag}.tmp"
    r = subprocess.run([cc, *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
    for o in objs:
        os.remove(o)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
