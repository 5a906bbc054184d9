"""Builds the CUDA library (sm_100a) in-tree with nvcc: csrc/*.cu -> lib/libvvs.so, and the CPython
entry points that marshal its calls: csrc/binding_native.c -> _native.<ABI of this interpreter>.so.

nvcc cross-compiles without a GPU.  Objects go to _build/ (not committed); the shared library
stays inside the package so that it travels with the source tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB_DIR = os.path.join(PKG, "lib")
LIB = os.path.join(LIB_DIR, "libvvs.so")
OBJ_DIR = os.path.join(PKG, "_build")
NATIVE_SRC = os.path.join(CSRC, "binding_native.c")
# named for this interpreter: another version does not take it for its own, neither to load nor as built already
NATIVE = os.path.join(PKG, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_UNTAGGED = os.path.join(PKG, "_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _newest_header() -> float:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs.append(os.path.join(ROOT, "include", "vvs.h"))
    return max(os.path.getmtime(h) for h in hs)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    os.makedirs(LIB_DIR, exist_ok=True)
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()
    srcs = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
    hdr_time = _newest_header()
    jobs = []
    for f in srcs:
        src = os.path.join(CSRC, f)
        obj = os.path.join(OBJ_DIR, f[:-3] + ".o")
        stale = force or not os.path.exists(obj) or \
            os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time)
        jobs.append((src, obj, stale))

    def compile_one(job):
        src, obj, stale = job
        if not stale:
            return ""
        cmd = [nvcc, *NVCC_FLAGS, *extra_flags, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        return r.stdout + r.stderr

    with ThreadPoolExecutor(max_workers=8) as ex:
        logs = list(ex.map(compile_one, jobs))
    if verbose:
        sys.stderr.write("".join(logs))
    objs = [j[1] for j in jobs]
    if force or any(j[2] for j in jobs) or not os.path.exists(LIB):
        cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    build_native(force)
    return LIB


def build_native(force: bool = False) -> str:
    """The extension module finds libvvs.so next to it (rpath), so both travel with the source tree."""
    newest = max(os.path.getmtime(p) for p in (NATIVE_SRC, os.path.join(ROOT, "include", "vvs.h")))
    if force or not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < newest:
        cmd = [os.environ.get("CC", "gcc"), "-shared", "-fPIC", "-O2", "-std=c11", "-Wall", "-I", sysconfig.get_paths()["include"],
               "-I", os.path.join(ROOT, "include"), NATIVE_SRC, "-o", NATIVE, "-L", LIB_DIR, "-l:libvvs.so",
               "-Wl,-rpath,$ORIGIN/lib"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"gcc failed for {NATIVE_SRC}:\n{r.stdout}\n{r.stderr}")
    if os.path.exists(NATIVE_UNTAGGED):       # of an earlier build: any interpreter without one of its own would load it
        os.remove(NATIVE_UNTAGGED)
    return NATIVE


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True,
                extra_flags=["-Xptxas", "-v"] if "--ptxas" in sys.argv else []))
