"""Builds libdraco.so (sm_100a) in-tree with nvcc.  No JIT, no cache outside the package."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libdraco.so")
# The CPython module of the calls that a training loop makes, named after the interpreter that it is built for: another one neither
# loads it nor takes it for up to date.
NATIVE = os.path.join(PKG, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))

SOURCES = ["draco_api.cu", "rep_kernels.cu", "cyc_encode.cu", "cyc_locate.cu", "cyc_onepass.cu", "cyc_recover.cu", "harness_kernels.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every translation unit for sm_100a and link libdraco.so; returns its path."""
    nvcc = _nvcc()
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(INCLUDE, "draco.h"), os.path.join(CSRC, "draco_internal.cuh")]
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src.replace(".cu", ".o"))
        if force or _stale(o, [s] + headers):
            cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        return r.stderr

    with ThreadPoolExecutor(max_workers=min(6, max(1, len(jobs)))) as ex:
        logs = list(ex.map(run, jobs))
    if verbose:
        sys.stderr.write("".join(logs))
    objs = [os.path.join(OBJ, s.replace(".cu", ".o")) for s in SOURCES]
    if force or jobs or _stale(LIB, objs):
        run([nvcc, "-shared", "-o", LIB] + objs + ["-lcudart"])
    src = os.path.join(CSRC, "native.cpp")
    python_include = sysconfig.get_paths()["include"]
    if force or _stale(NATIVE, [src, headers[0]]):
        if os.path.exists(os.path.join(python_include, "Python.h")):
            run([nvcc, "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", python_include, src,
                 "-o", NATIVE, "-L", PKG, "-Xlinker", "-l:libdraco.so", "-Xlinker", "-rpath=$ORIGIN"])
        else:
            sys.stderr.write(f"no Python.h in {python_include}: {os.path.basename(NATIVE)} is not built, ctypes makes its calls\n")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
