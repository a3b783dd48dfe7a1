"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libemo_b200.so")
SOURCES = ["emo_lib.cu", "emo_compile.cpp", "emo_flow_compile.cpp", "emo_spine_compile.cpp", "emo_slice_compile.cpp", "emo_contract.cpp", "emo_walk_compile.cpp", "emo_pack.cpp"]
HEADERS = ["emo_kernels.cuh", "emo_pass_staged.cuh", "emo_lane_layout.cuh", "emo_pass_lane.cuh", "emo_compile.h", "emo_flow.h", "emo_flow.cuh", "emo_spine.cuh", "emo_slice.h", "emo_contract.h", "emo_walk.h", "emo_walk.cuh", "emo_slice.cuh", "emo_intervals.cuh", "emo_model.cuh", "emo_generic.cuh",
           os.path.join("..", "..", "include", "emo.h")]


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(os.path.join(CSRC, f)) > t for f in SOURCES + HEADERS)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-o", tmp] + [os.path.join(CSRC, f) for f in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
