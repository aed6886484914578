"""Builds the CUDA library in-tree for sm_100a with nvcc (no GPU needed: nvcc cross-compiles)."""
from __future__ import annotations

import os
import subprocess
import sys

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libtandem_b200.so")
SOURCES = ["tandem_api.cu"]
EXT_SOURCE = os.path.join(CSRC, "standalone_py.cpp")          # Python entry to the stand-alone kernels
EXT_PATH = os.path.join(PKG_DIR, "_standalone.so")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC,-fvisibility=hidden", "-shared", "-cudart", "static"]


def _newest_source_mtime() -> float:
    newest = 0.0
    for root in (CSRC, os.path.join(os.path.dirname(PKG_DIR), "include")):
        for name in os.listdir(root):
            newest = max(newest, os.path.getmtime(os.path.join(root, name)))
    return newest


def _run(cmd, what: str, verbose: bool) -> None:
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
        raise RuntimeError(f"{cmd[0]} failed building {what}")
    if verbose:
        sys.stderr.write(proc.stderr)


def _build_extension(force: bool, verbose: bool) -> None:
    if not force and os.path.exists(EXT_PATH) and os.path.getmtime(EXT_PATH) >= _newest_source_mtime():
        return
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cpp_extension.CUDA_HOME or "/usr/local/cuda", "include")]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] + [f"-I{d}" for d in inc] + \
          [EXT_SOURCE, "-o", EXT_PATH, f"-L{lib}", "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10",
           f"-L{PKG_DIR}", "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN"]
    _run(cmd, EXT_PATH, verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles csrc/*.cu into libtandem_b200.so next to this file, and the Python entry to its stand-alone kernels;
    returns the library's path."""
    if force or not os.path.exists(LIB_PATH) or os.path.getmtime(LIB_PATH) < _newest_source_mtime():
        _run([os.environ.get("NVCC", "nvcc")] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) +
             [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB_PATH], LIB_PATH, verbose)
    _build_extension(force, verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
