"""In-tree build of libs4c.so (hand-written CUDA for sm_100a) with nvcc -- no torch types -- and of the native marshalling of the
eager calls (bind.cpp: torch tensors to the C ABI), with g++.  No JIT cache."""
from __future__ import annotations

import glob
import os
import re
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_HERE, "csrc")
_INC = os.path.join(os.path.dirname(_HERE), "include")
_LIB = os.path.join(_HERE, "libs4c.so")
_BIND_SRC = os.path.join(_CSRC, "bind.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall"]


def lib_path() -> str:
    return _LIB


def bind_path() -> str:
    """The native marshalling's binary.  It uses torch's C++ types, whose layout is that of one version, so its name says which torch
    and which Python it was built for: a binary of another version is not found (file times would not show the change)."""
    import torch

    version = re.sub(r"[^0-9A-Za-z]+", "_", f"{torch.__version__}_abi{int(torch._C._GLIBCXX_USE_CXX11_ABI)}")
    return os.path.join(_HERE, f"_bind.torch_{version}.{sysconfig.get_config_var('SOABI')}.so")


def sources():
    return sorted(glob.glob(os.path.join(_CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(_CSRC, "*.cuh")) + glob.glob(os.path.join(_CSRC, "*.h")) + \
        glob.glob(os.path.join(_INC, "*.h"))


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ for sm_100a and link libs4c.so next to this file."""
    deps = _deps()
    if not sources():
        raise RuntimeError("no CUDA sources found under " + _CSRC)
    newest = max(os.path.getmtime(p) for p in deps)
    if not force and os.path.exists(_LIB) and os.path.getmtime(_LIB) >= newest:
        _build_bind(force)
        return _LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    for src in sources():
        obj = os.path.splitext(src)[0] + ".o"
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, "-I", _INC, "-I", _CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd)))
    for src, p in procs:
        if p.wait() != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = _LIB + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-o", tmp, *objs, "-lcudart"], check=True)
    os.replace(tmp, _LIB)
    _build_bind(force)
    return _LIB


def _build_bind(force: bool = False) -> str:
    """Compile bind.cpp against torch's headers and libs4c.so (found next to it at run time)."""
    import torch

    path = bind_path()
    newest = max(os.path.getmtime(p) for p in [_BIND_SRC] + glob.glob(os.path.join(_INC, "*.h")))
    if not force and os.path.exists(path) and os.path.getmtime(path) >= newest:
        return path
    root = os.path.dirname(torch.__file__)
    lib = os.path.join(root, "lib")
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), _INC,
           sysconfig.get_paths()["include"], os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
    tmp = path + f".tmp{os.getpid()}"
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    *[f"-I{p}" for p in inc], _BIND_SRC, "-o", tmp, f"-L{_HERE}", "-l:libs4c.so", f"-L{lib}", "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10",
                    "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{lib}"], check=True)
    os.replace(tmp, path)
    return path
