"""Build the C-ABI CUDA library (libmixdq.so, nvcc for sm_100a) and its Python binding (_mixdq_native.so, g++) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmixdq.so")
BIND_SRC = os.path.join(CSRC, "bind.cpp")
BIND = os.path.join(HERE, "_mixdq_native.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _build_binding(force: bool) -> None:
    """The extension module links against libmixdq.so beside it; torch's libraries are found in the process, which has
    imported torch before it imports this package."""
    newest = max(os.path.getmtime(f) for f in (BIND_SRC, os.path.join(INCLUDE, "mixdq.h")))
    if not force and os.path.exists(BIND) and os.path.getmtime(BIND) >= newest:
        return
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-isystem", os.path.join(root, "include"),
                    "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
                    "-isystem", "/usr/local/cuda/include", "-I" + sysconfig.get_paths()["include"], BIND_SRC, "-o", BIND,
                    "-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda",
                    "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_library(force, verbose)
    _build_binding(force)
    return LIB


def _build_library(force: bool, verbose: bool) -> None:
    if not (force or _stale()):
        return
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    for src in sources():
        obj = os.path.join(HERE, "_build", os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
               "-Xcompiler", "-fPIC", "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if pr.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.run([nvcc, "-shared", "-cudart", "static", "-o", LIB] + objs, check=True)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
