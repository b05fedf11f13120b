"""Compiles the CUDA sources into ``libspf.so`` (sm_100a only) and the native part of the Python binding into
``_native.so``, both next to this file.

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
import sysconfig
import tempfile

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libspf.so")
NATIVE_SRC = os.path.join(CSRC, "python", "native.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_native.so")
NATIVE_FOR_PATH = NATIVE_PATH + ".for"       # the interpreter and the torch that _native.so was built against

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


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


def _running() -> str:
    import torch
    return f"python {sys.version_info.major}.{sys.version_info.minor}, torch {torch.__version__}"


def native_is_for() -> str:
    """What _native.so was built against, as _running() names it; empty if that is not known."""
    try:
        with open(NATIVE_FOR_PATH) as f:
            return f.read().strip()
    except OSError:
        return ""


def _native_is_stale() -> bool:
    return _older(NATIVE_PATH, [NATIVE_SRC, *glob.glob(os.path.join(ROOT, "include", "*.h"))]) or native_is_for() != _running()


def is_stale() -> bool:
    headers = glob.glob(os.path.join(ROOT, "include", "*.h"))
    return _older(LIB_PATH, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + headers) or _native_is_stale()


def _native_command() -> list:
    """g++ command for the binding's native part, against the headers and libraries of the installed torch."""
    import torch
    torch_dir = os.path.dirname(os.path.abspath(torch.__file__))
    include = [os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
               os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"), sysconfig.get_paths()["include"],
               os.path.join(ROOT, "include")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *[f"-I{d}" for d in include], NATIVE_SRC, "-o", NATIVE_PATH, f"-L{os.path.join(torch_dir, 'lib')}", "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", LIB_PATH, "-Wl,-rpath,$ORIGIN"]


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Builds libspf.so and _native.so if one of them is missing, older than its sources or (the latter) built against another
    torch or Python; returns the path of libspf.so."""
    if not force and not is_stale():
        return LIB_PATH
    include = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]

    def run(cmd):
        proc = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or proc.returncode != 0:
            sys.stderr.write(proc.stdout + proc.stderr)
        if proc.returncode != 0:
            raise RuntimeError("compilation failed: " + " ".join(cmd))
        return proc.stdout + proc.stderr

    with tempfile.TemporaryDirectory() as tmp:
        objects = [os.path.join(tmp, os.path.basename(src) + ".o") for src in sources()]
        with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 1) as pool:
            log = "".join(pool.map(lambda so: run([_nvcc(), *NVCC_FLAGS, *include, "-c", so[0], "-o", so[1]]), zip(sources(), objects)))
        run([_nvcc(), *NVCC_FLAGS, "--shared", "-o", LIB_PATH, "-Xlinker", "-soname=libspf.so", *objects])
    if force or _native_is_stale():
        run(_native_command())
        with open(NATIVE_FOR_PATH, "w") as f:
            f.write(_running() + "\n")
    with open(os.path.join(PKG_DIR, "libspf.ptxas.log"), "w") as f:
        f.write(log)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
