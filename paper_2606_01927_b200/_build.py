"""Builds ``libalbireo_sample.so`` (sm_100a only, nvcc) and ``_native.so`` (the binding's native half, g++) in-tree."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
_CSRC = os.path.join(_PKG, "csrc")
SOURCES = [os.path.join(_CSRC, "albireo_sample.cu")]
NATIVE_SOURCES = [os.path.join(_CSRC, "native_binding.cpp")]
INCLUDE = os.path.join(_ROOT, "include")
LIB_PATH = os.path.join(_PKG, "libalbireo_sample.so")
NATIVE_PATH = os.path.join(_PKG, "_native.so")


def nvcc_path() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def is_stale() -> bool:
    header = os.path.join(INCLUDE, "albireo_sample.h")
    parts = [os.path.join(_CSRC, f) for f in os.listdir(_CSRC) if f.endswith(".cuh")]
    return _older(LIB_PATH, SOURCES + parts + [header]) or _older(NATIVE_PATH, NATIVE_SOURCES + [header])


def _run(cmd, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(cmd[0] + " failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stdout + res.stderr)


def _build_native(verbose: bool) -> None:
    """The Python binding's native half (csrc/native_binding.cpp), against torch's headers and the CUDA library."""
    import torch
    from torch.utils import cpp_extension
    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda_home = os.path.dirname(os.path.dirname(nvcc_path()))
    tmp = NATIVE_PATH + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", INCLUDE, "-I", os.path.join(cuda_home, "include")]
    for inc in cpp_extension.include_paths() + [sysconfig.get_paths()["include"]]:
        cmd += ["-isystem", inc]
    cmd += ["-o", tmp] + NATIVE_SOURCES + ["-L", _PKG, "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN",
                                           "-L", libdir, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    _run(cmd, verbose)
    os.replace(tmp, NATIVE_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the CUDA library and the native half of the binding if they are missing or older than their sources."""
    if not force and not is_stale():
        return LIB_PATH
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    _run([nvcc_path(), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
          "-Xptxas", "-v", "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-soname=" + os.path.basename(LIB_PATH),
          "-I", INCLUDE, "-o", tmp] + SOURCES, verbose)
    os.replace(tmp, LIB_PATH)
    _build_native(verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
