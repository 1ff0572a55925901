"""Builds libnetmax.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnetmax.so")
SOURCES = ["netmax.cu", "netmax_fused.cu", "netmax_tiles_f32.cu", "netmax_tiles_bf16.cu", "netmax_pipe.cu", "netmax_policy.cpp", "netmax_policy_gpu.cu"]
HEADERS = ["netmax_policy_gpu_host.inc", "netmax_tile_instances.inc", "netmax_instances.h", "netmax_kernels.cuh", "netmax_plain.cuh", "netmax_tiles.cuh",
           "netmax_pipe.cuh", "netmax_rng.cuh", "netmax_fp64.cuh", "netmax_search.h", "netmax_policy.h", "netmax_bulk.h", os.path.join("..", "..", "include", "netmax.h")]
DEPS = SOURCES + HEADERS


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    built = os.path.getmtime(LIB)
    return any(os.path.getmtime(os.path.join(CSRC, d)) > built for d in DEPS)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile when the library is missing or older than a source; returns its path."""
    if not force and not is_stale():
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    flags = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-Xcompiler", "-fPIC,-O2,-pthread"]
    if verbose:
        flags += ["-Xptxas", "-v"]

    def run(args):
        return subprocess.run([_nvcc()] + flags + args, cwd=CSRC, capture_output=True, text=True)

    with tempfile.TemporaryDirectory() as objects, ThreadPoolExecutor(len(SOURCES)) as pool:  # a compiler for every source
        names = [os.path.join(objects, s + ".o") for s in SOURCES]
        done = list(pool.map(lambda job: run(["-c", os.path.join(CSRC, job[0]), "-o", job[1]]), zip(SOURCES, names)))
        if all(proc.returncode == 0 for proc in done):
            done.append(run(["-shared", "-o", tmp] + names))
    for proc in done:
        if verbose or proc.returncode != 0:
            sys.stderr.write(proc.stdout + proc.stderr)
        if proc.returncode != 0:
            raise RuntimeError("nvcc failed building libnetmax.so")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
