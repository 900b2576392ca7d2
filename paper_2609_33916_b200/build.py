"""Builds the CUDA library in-tree with nvcc for sm_100a (no GPU needed)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
import warnings
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(HERE, "libmoa_attn.so")
# (the suffix names the interpreter and its ABI: a tree built by one and used by another does not load the wrong module)
PYCALL = os.path.join(HERE, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--use_fast_math", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]
# the fp32 SIMT path is held to 1e-5 against the fp64 oracle: no fast-math there
NO_FAST_MATH = {"simt_kernels.cu"}


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    return "nvcc"


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    headers.append(os.path.abspath(__file__))
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            flags = [f for f in NVCC_FLAGS if not (f == "--use_fast_math" and os.path.basename(src) in NO_FAST_MATH)]
            if verbose:
                flags = flags + ["-Xptxas", "-v"]
            jobs.append([_nvcc()] + flags + ["-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {cmd[-3]}")

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        cmd = [_nvcc(), "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        run(cmd)
    build_pycall(force)
    return LIB


def build_pycall(force: bool = False) -> str | None:
    """The marshalling extension of binding.py (plain C, no CUDA).  None where it cannot be compiled (no compiler or no Python headers):
    the binding then marshals through ctypes."""
    untagged = os.path.join(HERE, "_pycall.so")
    if untagged != PYCALL and os.path.exists(untagged):      # (any interpreter would load it)
        os.remove(untagged)
    src = os.path.join(CSRC, "pycall.c")
    if force or _stale(PYCALL, [src]):
        include = sysconfig.get_paths()["include"]
        partial = f"{PYCALL}.{os.getpid()}"
        try:
            r = subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", include, src, "-o", partial],
                               capture_output=True, text=True)
        except OSError as e:
            warnings.warn(f"no C compiler for {src} ({e}): short calls take about 2 us longer")
            return None
        if r.returncode != 0:
            if os.path.exists(os.path.join(include, "Python.h")):
                raise RuntimeError(f"the compiler failed for {src}:\n{r.stderr}")
            warnings.warn(f"no Python headers for {src}: short calls take about 2 us longer")
            return None
        os.replace(partial, PYCALL)
    return PYCALL


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
