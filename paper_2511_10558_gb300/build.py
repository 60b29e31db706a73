"""Build libcarbox.so (sm_103a) in-tree with nvcc; no cmake, no torch extension.

``build()`` compiles the translation units in parallel and links them
into ``paper_2511_10558_gb300/lib/libcarbox.so``. It is skipped when the
library is newer than every source.
"""
from __future__ import annotations

import concurrent.futures
import os
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "lib", "libcarbox.so")
SOURCES = ["solve_fp64.cu", "solve_fp64_gm.cu", "solve_mixed.cu", "solve_mixed_gm.cu", "solve_fp64_rk.cu",
           "solve_mixed_rk.cu", "solve_fp64_gm_rk.cu", "solve_mixed_gm_rk.cu", "solve_fp64_narrow.cu", "solve_mixed_narrow.cu", "solve_fp64_mid.cu",
           "solve_mixed_mid.cu", "solve_fp64_two.cu", "solve_mixed_two.cu", "solve_fp64_gm_two.cu",
           "solve_mixed_gm_two.cu", "adjoint.cu", "plan.cu", "network.cpp",
           "capi.cpp", "esdirk.cpp", "noalloc.cu", "order.cu", "server.cpp", "peaks.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    files.append(os.path.abspath(__file__))
    return files


def source_hash() -> str:
    """Hash of the kernel sources (identifies the build a profile was taken on)."""
    import hashlib
    h = hashlib.sha256()
    for f in sorted(SOURCES) + ["internal.h", "solver_dev.cuh"]:
        h.update(open(os.path.join(CSRC, f), "rb").read())
    for f in sorted(os.listdir(INCLUDE)):
        h.update(open(os.path.join(INCLUDE, f), "rb").read())
    return h.hexdigest()[:16]


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB):
        newest = max(os.path.getmtime(f) for f in _deps())
        if os.path.getmtime(LIB) >= newest:
            return LIB
    os.makedirs(BUILD, exist_ok=True)
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    nvcc = _nvcc()
    common = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]

    def compile_one(src):
        obj = os.path.join(BUILD, src + ".o")
        cmd = [nvcc] + common + ["-c", os.path.join(CSRC, src), "-o", obj]
        if src.endswith(".cu"):
            cmd += ["-Xptxas", "-v"] if verbose else []
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{res.stderr}")
        if verbose and res.stderr:
            print(res.stderr)
        return obj

    with concurrent.futures.ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-cudart", "shared", "-o", tmp] + objs + \
        ["-Xlinker", "-rpath," + os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "lib64")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
