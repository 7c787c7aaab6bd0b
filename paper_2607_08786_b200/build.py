"""Builds ``libtl3.so`` in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import re
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libtl3.so")
SOURCES = ("tl3_host.cpp", "tl3_pack.cpp", "tl3_spmm.cu", "tl3_spmm_wide.cu", "tl3_encode.cu", "tl3_pack_device.cu", "tl3_convert.cu")
HEADERS = (os.path.join(CSRC, "tl3_internal.h"), os.path.join(CSRC, "tl3_device.cuh"), os.path.join(CSRC, "tl3_convert.cuh"), os.path.join(ROOT, "include", "tl3.h"))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + list(HEADERS)
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile and link the library if any source is newer than it; returns its path."""
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC,-Wall,-Wextra", "-Xptxas", "-v", "-shared",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        print(res.stdout)
        print(res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libtl3.so")
    # what tl3_copy_kernel counts on (tl3_spmm.cu) and launch bounds cannot ask for
    used = re.search(r"Compiling entry function '\w*tl3_copy_kernel\w*'.*?Used (\d+) registers", res.stdout + res.stderr, re.S)
    if used is None or int(used.group(1)) > 16:
        os.remove(LIB)
        raise RuntimeError(f"tl3_copy_kernel takes {used.group(1) if used else 'an unknown number of'} registers, not 16: it no longer fits beside a product")
    return LIB


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
