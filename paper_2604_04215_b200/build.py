"""Builds libdare.so (the C-ABI library) in-tree with nvcc for sm_100a.

    python -m paper_2604_04215_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The library links the static CUDA runtime and resolves the one driver
entry point it needs (tensor-map encoding) at run time, so it has no link-time dependency on libcuda.
The marshalling module beside it (marshal_path) is the Python module through which binding.py makes the calls of a
rollout's inner loop.  It reads torch's tensor objects, so it holds for one Python and one torch: both stand in its name,
and another torch neither loads it nor takes it for up to date.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdare.so")
SOURCES = ["api.cu", "lmhead.cu", "attn.cu", "select.cu", "gemm.cu", "gemm_few.cu", "layers.cu", "model.cu", "diffusion.cu", "backward.cu"]
HEADERS = ["ptx.cuh", "internal.h", os.path.join("..", "..", "include", "dare.h")]


def marshal_path() -> str:
    """Where the marshalling module for this Python and this torch is (or would be)."""
    import torch
    return os.path.join(HERE, f"_marshal-torch{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found")
    return cand


def _stale() -> bool:
    marshal = marshal_path()
    if not os.path.exists(LIB) or not os.path.exists(marshal):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(marshal))
    deps = [os.path.join(CSRC, s) for s in SOURCES + ["marshal.cpp"] + HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def _marshal_cmd() -> list:
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include"), sysconfig.get_paths()["include"]]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            *[f for d in inc for f in ("-isystem", d)], "-o", marshal_path(), os.path.join(CSRC, "marshal.cpp"),
            "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-ldl"]


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-DNDEBUG",
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    for what, c in (("libdare.so", cmd), (os.path.basename(marshal_path()), _marshal_cmd())):
        res = subprocess.run(c, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError(f"{c[0]} failed building {what}")
    return LIB


if __name__ == "__main__":
    path = build(force="--force" in sys.argv, verbose="--verbose" in sys.argv)
    print(path)
