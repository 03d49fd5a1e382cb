"""Builds libslkv.so (CUDA, sm_100a) and _slkv_call.so (the Python binding's call path) next to this file:  python -m paper_2508_15806_b200.build"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libslkv.so")
CALL = os.path.join(HERE, "_slkv_call.so")
SOURCES = ["slkv_api.cu", "slkv_alloc.cu", "slkv_score_simt.cu", "slkv_score_tc.cu", "slkv_score_pipe.cu", "slkv_select.cu", "slkv_select_cluster.cu", "slkv_select_cta.cu",
           "slkv_layer_tc.cu", "slkv_layer_fma.cu", "slkv_bound.cu", "slkv_noalloc.cu", "slkv_behavior.cu", "slkv_cp.cu"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    return "nvcc"


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALL))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "slkv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every source to an object file (in parallel) and links libslkv.so."""
    if not force and not needs_build():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    obj_dir = os.path.join(HERE, "build")
    os.makedirs(obj_dir, exist_ok=True)
    flags = ["-Xcompiler", "-fPIC", "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
             "-Xfatbin=-compress-all", "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        flags += ["-Xptxas", "-v"]

    def compile_one(src: str):
        obj = os.path.join(obj_dir, src.replace(".cu", ".o"))
        r = subprocess.run([_nvcc(), "-c", *flags, "-o", obj, os.path.join(CSRC, src)], capture_output=True, text=True)
        return obj, r

    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 4)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    for obj, r in results:
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("nvcc failed building libslkv.so")
        if verbose:
            sys.stderr.write(r.stdout + r.stderr)
    r = subprocess.run([_nvcc(), "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                        "-o", LIB, *[o for o, _ in results]], capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("nvcc failed linking libslkv.so")
    r = subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                        "-o", CALL, os.path.join(CSRC, "slkv_pycall.c")], capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("building _slkv_call.so failed")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
