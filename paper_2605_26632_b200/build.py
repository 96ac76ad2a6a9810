"""Builds ``liblynx.so`` (the C-ABI CUDA library, nvcc for sm_100a) and ``_lynx_calls.<tag>.so`` (the binding's per-layer
calls, a CPython extension on top of it) in-tree."""
from __future__ import annotations

import glob
import hashlib
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblynx.so")
HEADER = os.path.join(ROOT, "include", "lynx.h")
SOURCES = [os.path.join(CSRC, "lynx_api.cu")]
CALLS_SOURCES = [os.path.join(CSRC, "binding_calls.cpp")]
DEPS = [os.path.join(CSRC, f) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))] + [HEADER]
CALLS_DEPS = CALLS_SOURCES + [HEADER]


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def is_stale() -> bool:
    return _older(LIB, DEPS)


def calls_path() -> str:
    """The extension's file.  It inlines the layouts of CPython's and torch's objects and the library's C ABI, and a build for
    others may load and read wrong fields: its name says what it was built for, and no other file is ever loaded."""
    import torch

    h = hashlib.sha256(f"{torch.version.git_version} {int(torch._C._GLIBCXX_USE_CXX11_ABI)}".encode())
    for f in CALLS_DEPS:
        with open(f, "rb") as src:
            h.update(src.read())
    return os.path.join(HERE, f"_lynx_calls.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.{h.hexdigest()[:12]}.so")


def _nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def _run(cmd, target: str, verbose: bool):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{os.path.basename(cmd[0])} failed building {os.path.basename(target)}")


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
           "-Xcompiler", "-fPIC,-fvisibility=hidden", "-shared", "-o", tmp] + SOURCES + ["-lcudart"]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    _run(cmd, LIB, verbose)
    os.replace(tmp, LIB)
    return LIB


def build_calls(force: bool = False, verbose: bool = False) -> str:
    """Needs liblynx.so, and torch's headers and libraries as installed.  -> calls_path()"""
    path = calls_path()
    if not force and os.path.exists(path):
        return path
    import torch

    torch_dir = os.path.dirname(os.path.abspath(torch.__file__))
    cuda_include = os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")
    tmp = path + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I" + sysconfig.get_paths()["include"], "-isystem", os.path.join(torch_dir, "include"),
           "-isystem", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), "-isystem", cuda_include]
    cmd += CALLS_SOURCES + ["-o", tmp, "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
                            "-lc10_cuda", "-L" + HERE, "-l:liblynx.so", "-Wl,-rpath,$ORIGIN"]
    _run(cmd, path, verbose)
    os.replace(tmp, path)
    for old in glob.glob(glob.escape(path.rsplit(".", 2)[0]) + ".*.so"):  # of other sources
        if old != path:
            os.remove(old)
    return path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_calls(force="--force" in sys.argv, verbose="-v" in sys.argv))
