"""Build libvlb.so in-tree for sm_103a (GB300) with nvcc.

Each CUDA translation unit is compiled in parallel, then linked into one shared library with
the CUDA runtime linked statically (no torch types cross the C ABI).  Usage:

    python -m paper_1904_10070_gb300.build [--verbose-ptxas]
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libvlb.so")
SOURCES = ["vlb_stage.cu", "vlb_direct.cu", "vlb_axi.cu", "vlb_aux.cu", "vlb_capi.cu", "vlb_noalloc.cu", "vlb_conv.cu", "vlb_conv_tc.cu", "vlb_surrogate.cu",
           "vlb_surrogate_api.cu", "vlb_chsolve.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr"]


def nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def stage_tag() -> str:
    """64-bit hash of the sources of the packed FP32 stage: the key of kept autotune choices and of measured traffic."""
    h = hashlib.sha256()
    for name in ("vlb_stage.cu", "vlb_node.cuh", "vlb_internal.cuh"):
        with open(os.path.join(CSRC, name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def _compile(src: str, verbose_ptxas: bool) -> str:
    obj = os.path.join(BUILD, src.replace(".cu", ".o"))
    cmd = [nvcc(), *ARCH, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
    if src == "vlb_capi.cu":
        cmd.append(f"-DVLB_ENSEMBLE_TAG=0x{stage_tag()}ull")
    if verbose_ptxas:
        cmd += ["-Xptxas", "-v"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{res.stdout}\n{res.stderr}")
    if verbose_ptxas:
        sys.stderr.write(res.stderr)
    return obj


def build(verbose_ptxas: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose_ptxas), SOURCES))
    tmp = LIB + ".tmp"
    # only the C ABI (vlb_*) is exported; the kernels' C++ symbols stay internal to the library
    vmap = os.path.join(CSRC, "libvlb.map")
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "static", "-Xlinker", f"--version-script={vmap}", "-o", tmp, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose_ptxas="--verbose-ptxas" in sys.argv))
