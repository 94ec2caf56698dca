"""In-tree build of the CUDA library: nvcc -> paper_2608_08081_b200/libisoquant.so (sm_100a only)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libisoquant.so")
SOURCES = ["iq_api.cu", "iq_quantize.cu", "iq_append_bulk.cu", "iq_decode.cu", "iq_decode_b2.cu", "iq_decode_b3.cu", "iq_decode_b4.cu", "iq_combine.cu",
           "iq_static.cu", "iq_reconstruct.cu", "iq_reconstruct_tile.cu"]
HEADERS = ["iq_common.cuh", "iq_decode_common.cuh", "iq_decode_kernel.cuh", "iq_quantize_common.cuh", "iq_append_row.cuh", "iq_tile_mma.cuh", "iq_format.cuh",
           "iq_kernels.h", os.path.join("..", "..", "include", "isoquant.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-t", "0",
              "-Xcompiler", "-fPIC", "-shared"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    extra = os.environ.get("IQ_NVCC_EXTRA", "").split()
    cmd = [_nvcc()] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(r.stderr)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + r.stdout + r.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
