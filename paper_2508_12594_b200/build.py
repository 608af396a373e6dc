"""Builds libflare.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the Python extension that marshals torch
tensors for it (g++).

``python -m paper_2508_12594_b200.build`` or ``build()``.  nvcc cross-compiles without a GPU.  The translation units are
compiled side by side; an object is compiled again only when its source or a file it includes has changed.
"""
from __future__ import annotations

import concurrent.futures
import os
import re
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(_HERE, "..", "include")
OBJ = os.path.join(_HERE, "_build")
LIB = os.path.join(_HERE, "libflare.so")
BINDING_SRC = os.path.join(CSRC, "flare_binding.cpp")
BINDING = os.path.join(_HERE, "_binding.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-cudart", "static", "-Xptxas", "-v",
]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps(path: str, seen=None):
    """The file and everything of this repository it includes."""
    seen = set() if seen is None else seen
    path = os.path.normpath(path)
    if path in seen or not os.path.exists(path):
        return seen
    seen.add(path)
    with open(path) as f:
        for name in re.findall(r'^#include "([^"]+)"', f.read(), flags=re.M):
            _deps(os.path.join(os.path.dirname(path), name), seen)
    return seen


def _object(src: str) -> str:
    return os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")


def _newer(target: str, deps) -> bool:
    return os.path.exists(target) and all(os.path.getmtime(d) <= os.path.getmtime(target) for d in deps)


def _compile(src: str):
    obj = _object(src)
    tmp = obj + f".{os.getpid()}.tmp.o"
    res = subprocess.run([NVCC] + FLAGS + ["-c", "-o", tmp, src], capture_output=True, text=True)
    if res.returncode == 0:
        with open(obj[:-2] + ".ptxas.txt", "w") as f:
            f.write(res.stderr)
        os.replace(tmp, obj)
    return src, res


def _compile_binding(src: str):
    """The marshalling extension: plain C++ against this interpreter's and torch's headers."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    tmp = BINDING + f".{os.getpid()}.tmp"
    includes = [f"-I{p}" for p in cpp_extension.include_paths()] + [f"-I{sysconfig.get_paths()['include']}", "-I/usr/local/cuda/include"]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           *includes, "-o", tmp, src, *[f"-L{p}" for p in cpp_extension.library_paths()],
           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode == 0:
        os.replace(tmp, BINDING)
    return src, res


def _stale() -> bool:
    deps = set()
    for s in sources():
        _deps(s, deps)
    return not (_newer(LIB, deps) and _newer(BINDING, _deps(BINDING_SRC)))


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or _stale()):
        return LIB
    os.makedirs(OBJ, exist_ok=True)
    todo = [s for s in sources() if force or not _newer(_object(s), _deps(s))]
    todo.sort(key=os.path.getsize, reverse=True)
    if force or not _newer(BINDING, _deps(BINDING_SRC)):
        todo.append(BINDING_SRC)
    with concurrent.futures.ThreadPoolExecutor(max_workers=max(1, os.cpu_count() or 1)) as pool:
        for src, res in pool.map(lambda s: _compile_binding(s) if s == BINDING_SRC else _compile(s), todo):
            if verbose or res.returncode != 0:
                sys.stderr.write(res.stdout + res.stderr)
            if res.returncode != 0:
                raise RuntimeError(f"failed compiling {os.path.basename(src)}")
    tmp = LIB + f".{os.getpid()}.tmp"
    res = subprocess.run([NVCC] + FLAGS[:2] + ["--shared", "-Xcompiler", "-fPIC", "-cudart", "static", "-o", tmp] +
                         [_object(s) for s in sources()], capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed linking libflare.so")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
