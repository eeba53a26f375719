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
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newest(files) -> float:
    return max(os.path.getmtime(f) for f in files)


def _fresh(target: str, files) -> bool:
    return os.path.exists(target) and os.path.getmtime(target) >= _newest(files)


def _headers():
    return [f for pattern in (os.path.join(CSRC, "*.cuh"), os.path.join(CSRC, "*.h"), os.path.join(INCLUDE, "*.h"))
            for f in glob.glob(pattern)]


def _build_binding(force: bool) -> None:
    """The extension module links against libmixdq.so beside it; torch's libraries are found in the process, which has
    imported torch before it imports this package.  What it was compiled against is compiled into it."""
    import sysconfig

    import torch
    built_for = f"_mixdq_native for torch {torch.__version__}, Python {sys.version_info.major}.{sys.version_info.minor}"
    if not force and _fresh(BIND, (BIND_SRC, os.path.join(CSRC, "unlocked.h"), os.path.join(INCLUDE, "mixdq.h"))):
        with open(BIND, "rb") as f:
            if built_for.encode() + b"\0" in f.read():
                return
    root = os.path.dirname(torch.__file__)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-isystem", os.path.join(root, "include"),
                    "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
                    "-isystem", "/usr/local/cuda/include", "-I" + sysconfig.get_paths()["include"],
                    f'-DMIXDQ_BUILT_FOR="{built_for}"', BIND_SRC, "-o", BIND,
                    "-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda",
                    "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_library(force, verbose)
    _build_binding(force)
    return LIB


def _build_library(force: bool, verbose: bool) -> None:
    if force or not _fresh(LIB, sources() + _headers()):
        subprocess.run([NVCC, "-shared", "-cudart", "static", "-o", LIB] + objects(force, verbose), check=True)


def objects(force: bool = False, verbose: bool = False) -> list:
    """The library's object files; those older than their source or any header are compiled."""
    objs = []
    procs = []
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    for src in sources():
        obj = os.path.join(HERE, "_build", os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if not force and _fresh(obj, [src] + _headers()):
            continue
        cmd = [NVCC, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
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
    return objs


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
