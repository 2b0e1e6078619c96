"""Builds libtokenscale.so (CUDA kernels + C ABI) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libtokenscale.so")
SOURCES = ["ts_host.cpp", "ts_layer.cpp", "ts_kernels.cu", "ts_decode.cu", "ts_mixed.cu", "ts_gemm.cu", "ts_layer_kernels.cu"]
HEADERS = [os.path.join(CSRC, "ts_internal.h"), os.path.join(CSRC, "ts_tma.h"), os.path.join(CSRC, "ts_ptx.h"), os.path.join(CSRC, "ts_tc.h"), os.path.join(CSRC, "ts_units.h"), os.path.join(CSRC, "ts_decode_body.h"),
           os.path.join(PKG_DIR, "..", "include", "tokenscale.h")]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile when the library is missing or older than its sources; returns its path."""
    if not force and not is_stale():
        return LIB_PATH
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-o", tmp] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
