"""Build ``libccm_gb300.so`` in-tree with nvcc for sm_103a.

Each CUDA translation unit (the search kernels: one per E) is compiled in parallel (one ``-gencode`` for
sm_103a, ``-lineinfo``, IEEE FP32: no fast-math, so ``sqrtf``, division and
``expf`` keep their documented accuracy) and linked with the static CUDA
runtime into one shared library exporting the C ABI of include/ccm.h.
"""

from __future__ import annotations

import concurrent.futures as cf
import hashlib
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libccm_gb300.so")
# (source, E): the search kernels are compiled once per embedding dimension, in parallel
SOURCES = [(name, e) for e in range(10, 0, -1) for name in ("knn_fused.cu", "table_build.cu", "knn_scan.cu")] + [
    (name, 0) for name in ("table.cu", "runtime.cu", "sampler.cu", "knn_dispatch.cu", "plain.cu",
                           "noalloc.cu", "order.cu", "convergence.cu")]
HEADERS = [os.path.join(CSRC, name) for name in (
    "ccm_internal.h", "moments.cuh", "bits.cuh", "row_walk.cuh", "launch.cuh")] + [
    os.path.join(INCLUDE, "ccm.h")]
# the search kernels that the autotuner chooses between: its cached choices carry their hash
TUNED = [os.path.join(CSRC, name) for name in ("knn_fused.cu", "ccm_internal.h", "moments.cuh")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _revision() -> str:
    h = hashlib.sha256()
    for path in TUNED:
        with open(path, "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def _compile(src: str, E: int, verbose: bool) -> str:
    obj = os.path.join(BUILD, os.path.splitext(src)[0] + (f"_e{E}" if E else "") + ".o")
    deps = [os.path.join(CSRC, src), *HEADERS, *(TUNED if src == "runtime.cu" else [])]
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(d) for d in deps):
        return obj
    cmd = [_nvcc(), *ARCH, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
           *([f"-DCCM_E={E}"] if E else []),
           *([f'-DCCM_KERNEL_REVISION="{_revision()}"'] if src == "runtime.cu" else []),
           *os.environ.get("CCM_EXTRA_NVCC_FLAGS", "").split(),
           "-I", INCLUDE, "-I", CSRC, "-c", os.path.join(CSRC, src), "-o", obj + ".tmp"]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    if verbose:
        sys.stderr.write(r.stderr)
    os.replace(obj + ".tmp", obj)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile (if stale) and link the library; returns its path."""
    os.makedirs(BUILD, exist_ok=True)
    if force:
        for f in os.listdir(BUILD):
            os.remove(os.path.join(BUILD, f))
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(lambda s: _compile(*s, verbose), SOURCES))
    if force or not os.path.exists(LIB) or os.path.getmtime(LIB) < max(os.path.getmtime(o) for o in objs):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [_nvcc(), *ARCH, "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", *objs,
               "-o", tmp]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
