"""Builds ``librac.so`` (the C-ABI library of CUDA kernels) in-tree with nvcc for sm_100a, and ``_native`` (the extension
module that marshals its calls) with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librac.so")
NATIVE = os.path.join(HERE, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_SOURCES = ["rac_py.cpp", os.path.join("..", "..", "include", "rac.h")]
SOURCES = ["rac_codec.cu", "rac_codec_dyn.cu", "rac_calib.cu", "rac_match.cu"]
HEADERS = ["rac_common.cuh", "rac_codec_dev.cuh", os.path.join("..", "..", "include", "rac.h")]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--threads", "0", "-Xptxas", "-v",
]


def _stale(target: str, sources) -> bool:
    return not os.path.exists(target) or os.path.getmtime(target) < max(os.path.getmtime(os.path.join(CSRC, f)) for f in sources)


def _compile(target: str, cmd, verbose: bool) -> None:
    """Run a compiler that writes to ``target`` + a suffix of this process, and put the result in place."""
    tmp = target + f".tmp{os.getpid()}"
    try:
        res = subprocess.run([tmp if c is None else c for c in cmd], capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("failed: " + " ".join(c or target for c in cmd))
        os.replace(tmp, target)
    finally:
        if os.path.exists(tmp):     # a failed or interrupted build leaves nothing behind
            os.remove(tmp)


def build_native(force: bool = False, verbose: bool = False) -> str:
    """The extension module; needs librac.so to link against, which it finds beside itself at run time."""
    if force or _stale(NATIVE, NATIVE_SOURCES):
        import torch
        from torch.utils import cpp_extension
        inc = [f"-I{p}" for p in cpp_extension.include_paths("cuda")] + [f"-I{sysconfig.get_paths()['include']}"]
        lib = [f"-L{p}" for p in cpp_extension.library_paths("cuda")]
        _compile(NATIVE, [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
                          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *inc, "-o", None,
                          os.path.join(CSRC, "rac_py.cpp"), *lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
                          "-lc10_cuda", f"-L{HERE}", "-l:librac.so", "-Wl,-rpath,$ORIGIN"], verbose)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is missing or older than its sources.  Returns the library path."""
    if force or _stale(LIB, SOURCES + HEADERS):
        _compile(LIB, [os.environ.get("NVCC", "nvcc"), *NVCC_FLAGS, "-o", None, *[os.path.join(CSRC, s) for s in SOURCES]], verbose)
    build_native(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
