"""Builds, in-tree and without a JIT cache, ``libattnw.so`` (nvcc, sm_100a) and ``_attnw_torch`` (host compiler): the
extension module that takes torch tensors to the library's C ABI without Python in between."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libattnw.so")
SOURCES = [os.path.join(_CSRC, "attnw_api.cu")]
_DEPS = [os.path.join(_CSRC, f) for f in sorted(os.listdir(_CSRC))] + [
    os.path.join(os.path.dirname(_PKG), "include", "attnw.h")]
EXT_PATH = os.path.join(_PKG, "_attnw_torch.so")
EXT_SOURCE = os.path.join(_CSRC, "torch_calls.cpp")
_DEPS.remove(EXT_SOURCE)


def nvcc_path() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; it is needed to build libattnw.so")


def nvcc_command(out: str, verbose_ptxas: bool = False, defines: tuple[str, ...] = ()) -> list[str]:
    cmd = [nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-o", out, *SOURCES]
    if verbose_ptxas:
        cmd[1:1] = ["-Xptxas", "-v"]
    for d in defines:
        cmd.insert(1, "-D" + d)
    return cmd


def built_for() -> str:
    """What ``_attnw_torch`` is bound to: the C++ interface of one torch and the C interface of one Python.  The module carries it."""
    import torch
    return f"attnw for torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def ext_command(out: str) -> list[str]:
    import torch
    from torch.utils import cpp_extension
    torch_lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda_home = os.path.dirname(os.path.dirname(nvcc_path()))
    includes = [sysconfig.get_paths()["include"], *cpp_extension.include_paths(), os.path.join(cuda_home, "include")]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DATTNW_BUILT_FOR="{built_for()}"',
            *["-isystem" + i for i in includes],
            "-o", out, EXT_SOURCE, "-L" + _PKG, "-l:" + os.path.basename(LIB_PATH), "-L" + torch_lib, "-ltorch_python",
            "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"]


def _older(target: str, deps: list[str]) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def is_stale() -> bool:
    return _older(LIB_PATH, _DEPS)


def ext_is_stale() -> bool:
    if _older(EXT_PATH, [EXT_SOURCE, os.path.join(os.path.dirname(_PKG), "include", "attnw.h")]):
        return True
    with open(EXT_PATH, "rb") as f:
        return built_for().encode() + b"\0" not in f.read()


def _compile(cmd: list[str], tmp: str, target: str) -> str:
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed:\n" + proc.stdout + proc.stderr)
    os.replace(tmp, target)
    return proc.stderr


def build_extension(force: bool = False) -> str:
    """Compile ``_attnw_torch`` if it is missing, older than its source or the C header, or built for another torch or Python;
    returns its path."""
    if force or ext_is_stale():
        tmp = EXT_PATH + f".tmp{os.getpid()}"
        _compile(ext_command(tmp), tmp, EXT_PATH)
    return EXT_PATH


def build_library(force: bool = False, verbose_ptxas: bool = False, defines: tuple[str, ...] = (),
                  out: str | None = None) -> str:
    """Compile if the library is missing or older than its sources; returns its path.  `defines` and `out` build a
    variant beside the product library (the instrumented build of timeline.py); the product library has none."""
    target = out or LIB_PATH
    if defines and out is None:
        raise ValueError("a build with extra definitions needs its own output path")
    if force or out is not None or is_stale():
        tmp = target + f".tmp{os.getpid()}"
        messages = _compile(nvcc_command(tmp, verbose_ptxas, defines), tmp, target)
        if verbose_ptxas:
            print(messages)
    if out is None:
        build_extension(force)
    return target


if __name__ == "__main__":
    import sys
    print(build_library(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv))
