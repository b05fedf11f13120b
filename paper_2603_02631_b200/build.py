"""Compiles the CUDA sources into ``libspf.so`` next to this file (sm_100a only).

Usage: ``python -m paper_2603_02631_b200.build [--force] [--verbose]``.
nvcc cross-compiles without a GPU, so this also runs on a CPU-only machine.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import shutil
import subprocess
import sys
import tempfile

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libspf.so")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC,-fvisibility=hidden", "-Xptxas", "-v",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; set NVCC or add it to PATH")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Builds libspf.so if it is missing or older than its sources; returns its path."""
    if not force and not is_stale():
        return LIB_PATH
    include = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]

    def run(cmd):
        proc = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or proc.returncode != 0:
            sys.stderr.write(proc.stdout + proc.stderr)
        if proc.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
        return proc.stdout + proc.stderr

    with tempfile.TemporaryDirectory() as tmp:
        objects = [os.path.join(tmp, os.path.basename(src) + ".o") for src in sources()]
        with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 1) as pool:
            log = "".join(pool.map(lambda so: run([_nvcc(), *NVCC_FLAGS, *include, "-c", so[0], "-o", so[1]]), zip(sources(), objects)))
        run([_nvcc(), *NVCC_FLAGS, "--shared", "-o", LIB_PATH, *objects])
    with open(os.path.join(PKG_DIR, "libspf.ptxas.log"), "w") as f:
        f.write(log)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
