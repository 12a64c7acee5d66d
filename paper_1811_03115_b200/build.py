"""Compile the CUDA library in-tree (nvcc, sm_100a only)."""
from __future__ import annotations

import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libbpd.so")
OBJ_DIR = os.path.join(HERE, "build")
SOURCES = ["layer_stack.cu", "layer_stack_512.cu", "layer_stack_256.cu", "fused_layer.cu", "gemm_tc.cu", "attention.cu", "bpd.cu", "noalloc.cu"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(HERE, "..", "include", "bpd.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Build ``libbpd.so`` next to this file if it is missing or older than its sources."""
    if not force and not _stale():
        return LIB_PATH
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
    if verbose:
        flags += ["-Xptxas", "-v"]
    os.makedirs(OBJ_DIR, exist_ok=True)
    objs = [os.path.join(OBJ_DIR, s[:-3] + ".o") for s in SOURCES]
    # one nvcc per translation unit, side by side
    procs = [(s, subprocess.Popen([_nvcc(), *flags, "-c", "-o", o, os.path.join(CSRC, s)], stdout=subprocess.PIPE,
                                  stderr=subprocess.STDOUT, text=True)) for s, o in zip(SOURCES, objs)]
    for name, proc in procs:
        out, _ = proc.communicate()
        if proc.returncode != 0:
            for _, other in procs:
                other.kill()
            raise RuntimeError(f"nvcc failed on {name}:\n{out}")
        if verbose:
            print(out)
    link = subprocess.run([_nvcc(), *flags, "-shared", "-o", LIB_PATH, *objs], capture_output=True, text=True)
    if link.returncode != 0:
        raise RuntimeError("linking failed:\n" + link.stdout + link.stderr)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
