"""Builds, in-tree, libmixkv.so (the C-ABI CUDA library, nvcc for sm_100a) and _mixkv_host.so (the native
half of the Python binding, the host compiler against torch's headers)."""
from __future__ import annotations

import glob
import hashlib
import importlib.util
import os
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(os.path.dirname(PKG), "include")
LIB = os.path.join(PKG, "libmixkv.so")
HOST_SRC = os.path.join(CSRC, "host", "host_binding.cpp")
HOST_LIB = os.path.join(PKG, "_mixkv_host.so")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--threads", "0", "-Xcompiler", "-fPIC", "-shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _headers():
    return (glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) +
            glob.glob(os.path.join(INCLUDE, "*.h")))


def is_stale() -> bool:
    return _older(LIB, sources() + _headers())


def _torch_root() -> str:
    return os.path.dirname(importlib.util.find_spec("torch").origin)   # (found, not imported)


def host_tag() -> str:
    """What _mixkv_host.so is bound to: this torch build's C++ interface and this Python's ABI.  The module
    carries it as a string."""
    with open(os.path.join(_torch_root(), "version.py"), "rb") as f:
        torch_build = hashlib.sha256(f.read()).hexdigest()[:16]
    return f"mixkv-host torch-{torch_build} {sysconfig.get_config_var('SOABI')}"


def host_matches(path: str = HOST_LIB) -> bool:
    """Whether the module was built for the torch and the Python in use (loading another one may crash)."""
    with open(path, "rb") as f:
        return host_tag().encode() + b"\0" in f.read()


def host_is_stale() -> bool:
    return _older(HOST_LIB, [HOST_SRC, os.path.join(CSRC, "internal_api.h"),
                             os.path.join(INCLUDE, "mixkv.h")]) or not host_matches()


def _host_command(out: str):
    import torch
    root = _torch_root()
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [INCLUDE, os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DMIXKV_HOST_TAG="{host_tag()}"',
            *[f"-I{d}" for d in inc], "-o", out, HOST_SRC, f"-L{os.path.join(root, 'lib')}",
            "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-lc10", "-lc10_cuda", "-ldl"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source of the package into libmixkv.so and the native binding into
    _mixkv_host.so (no GPU needed)."""
    jobs = []
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc, *NVCC_FLAGS, f"-I{INCLUDE}", f"-I{CSRC}", "-o", tmp, *sources()]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        jobs.append((cmd, tmp, LIB))
    if force or host_is_stale():
        tmp = HOST_LIB + f".tmp{os.getpid()}"
        jobs.append((_host_command(tmp), tmp, HOST_LIB))
    running = [(subprocess.Popen(cmd), cmd, tmp, lib) for cmd, tmp, lib in jobs]   # side by side
    failed = None
    for proc, cmd, tmp, lib in running:
        if proc.wait() != 0:
            failed = subprocess.CalledProcessError(proc.returncode, cmd)
        else:
            os.replace(tmp, lib)
    if failed:
        raise failed
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
