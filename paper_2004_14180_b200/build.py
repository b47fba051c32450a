"""Builds paper_2004_14180_b200/libqadam.so from csrc/ with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libqadam.so")
SOURCES = [os.path.join(CSRC, "qadam_api.cu"), os.path.join(CSRC, "qadam_noalloc.cu")]
HEADERS = [os.path.join(CSRC, "qadam_device.cuh"), os.path.join(CSRC, "qadam_kernels.cuh"),
           os.path.join(CSRC, "qadam_server_pipe.cuh"),
           os.path.join(CSRC, "qadam_worker_resident.cuh"), os.path.join(CSRC, "qadam_worker_stream.cuh"),
           os.path.join(CSRC, "qadam_host.h"),
           os.path.join(_ROOT, "include", "qadam.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    # IEEE arithmetic everywhere: no FMA contraction, exact division and root, subnormals kept
    "--fmad=false", "--prec-div=true", "--prec-sqrt=true", "--ftz=false",
    "-Xcompiler", "-fPIC", "-shared",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in SOURCES + HEADERS)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    cmd = [_nvcc()] + NVCC_FLAGS + ["-I", os.path.join(_ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-o", LIB] + SOURCES
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
