"""Compile the CUDA sources into paper_2504_03702_b200/libpreserve_b200.so for sm_100a.

nvcc cross-compiles without a GPU.  The library is built in-tree so that it travels with
the source tree; nothing is cached elsewhere.  Each source is compiled by a process of its own (the router's
instantiations alone take six minutes one after another); its object and what ptxas says of its kernels
(registers, stack, spills) go to _build/.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libpreserve_b200.so")
OBJECTS = os.path.join(HERE, "_build")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def report(source: str) -> str:
    """Where ptxas' report on a source's kernels is kept."""
    return _object(source)[:-2] + ".ptxas.txt"


def _object(source: str) -> str:
    return os.path.join(OBJECTS, os.path.basename(source)[:-3] + ".o")


def _older(made: str, deps) -> bool:
    return not os.path.exists(made) or any(os.path.getmtime(d) > os.path.getmtime(made) for d in deps)


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]


def _compile(source: str) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "--fmad=false",  # the router score is defined with separately rounded operations
           "-Xcompiler", "-fPIC", "-Xptxas", "-v", "-I", INCLUDE, "-I", CSRC, "-c", "-o", _object(source), source]
    done = subprocess.run(cmd, stderr=subprocess.PIPE, text=True)
    if done.returncode != 0:
        sys.stderr.write(done.stderr)
        raise subprocess.CalledProcessError(done.returncode, cmd)
    with open(report(source), "w") as f:
        f.write(done.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _older(LIB, sources() + _headers()):
        return LIB
    os.makedirs(OBJECTS, exist_ok=True)
    todo = [s for s in sources() if force or _older(report(s), [s] + _headers())]
    todo.sort(key=lambda s: "route_summary_" not in s)      # (the long ones first)
    with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 1) as pool:
        list(pool.map(_compile, todo))
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared", "-o", LIB]
                   + [_object(s) for s in sources()], check=True)
    if verbose:
        for s in sources():
            print(open(report(s)).read(), end="")
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
