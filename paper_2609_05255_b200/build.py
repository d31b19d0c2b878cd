"""Build libgs_b200.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libgs_b200.so")
SOURCES = ["gs_api.cu", "gs_preprocess.cu", "gs_sort.cu", "gs_depth_sort.cu", "gs_bin_cluster.cu", "gs_blend.cu", "gs_adam.cu", "gs_prepass.cu",
           "gs_decoder_variants.cu"]
HEADERS = [os.path.join(CSRC, h) for h in ("gs_device.cuh", "gs_bin.cuh", "gs_mlp_mma.cuh", "gs_decoder_tc.cuh", "gs_tcgen05.cuh", "gs_variants_tc.cuh")] + [os.path.join(_ROOT, "include", "gs.h")]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
