"""Builds the CUDA library in-tree: csrc/*.cu, *.cpp -> libaet_b200.so (sm_100a)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libaet_b200.so")
SOURCES = ["aet_api.cu", "aet_schedule.cpp", "lr_kernel.cu", "lr_chain_kernel.cu", "lr_relay_kernel.cu", "lr_block_kernel.cu", "mlp_kernel.cu", "mlp_mma_kernel.cu", "mlp_wide_kernel.cu", "mlp_tc_kernel.cu", "cnn_kernel.cu", "cnn_mma_kernel.cu", "agg_kernel.cu", "no_alloc.cu",
           "device_info.cu"]


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "aet.h"))
    return _newest(deps) > os.path.getmtime(LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found: cannot build libaet_b200.so")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "--threads", "4", "-Xcompiler", "-fPIC,-O3,-pthread", "-shared", "-cudart", "static",
           "-x", "cu"] + [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB + ".tmp", "-lpthread"]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    os.replace(LIB + ".tmp", LIB)
    if verbose:
        sys.stderr.write(res.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
