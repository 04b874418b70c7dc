"""Builds the native code in-tree: nvcc for sm_100a -> libllvq.so, and the host compiler -> _native.so (the torch
binding of its calls)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
HEADER = os.path.join(HERE, "..", "include", "llvq.h")
SOURCES = ["llvq_api.cu", "llvq_batch.cu", "llvq_expand.cu", "llvq_gemv.cu", "llvq_rotate.cu", "llvq_tables.cpp", "llvq_unrank.cpp"]
LIB = os.path.join(HERE, "libllvq.so")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared"]
BINDING_SOURCE = "llvq_torch.cpp"
BINDING = os.path.join(HERE, "_native.so")


def _tool(name: str, fallback: str) -> str:
    exe = shutil.which(name) or fallback
    if not os.path.exists(exe):
        raise RuntimeError(f"{name} not found: the native code cannot be built")
    return exe


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, target: str) -> None:
    tmp = target + f".tmp{os.getpid()}"
    subprocess.check_call([*cmd, "-o", tmp])
    os.replace(tmp, target)


def binding_tag() -> str:
    """The torch and the Python that _native.so is built for: it holds the layouts of both, so it must run under no other."""
    import torch

    return f"torch {torch.__version__} {torch.version.git_version}, {sysconfig.get_config_var('SOABI')}"


def _built_for_another() -> bool:
    """Whether _native.so lacks the tag of the torch and the Python that run now."""
    with open(BINDING, "rb") as f:
        return binding_tag().encode() + b"\0" not in f.read()


def _build_binding() -> None:
    import torch

    root = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.path.dirname(os.path.dirname(_tool("nvcc", "/usr/local/cuda/bin/nvcc"))), "include")
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), cuda,
               sysconfig.get_paths()["include"]]
    _run([_tool("g++", "/usr/bin/g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f'-DLLVQ_BUILT_FOR="{binding_tag()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          *["-isystem" + d for d in include], os.path.join(CSRC, BINDING_SOURCE), "-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda",
          "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"], BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    own = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != BINDING_SOURCE] + [HEADER]
    if force or _stale(LIB, own):
        _run([_tool("nvcc", "/usr/local/cuda/bin/nvcc"), *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []),
              *[os.path.join(CSRC, s) for s in SOURCES]], LIB)
    if force or _stale(BINDING, [os.path.join(CSRC, BINDING_SOURCE), HEADER]) or _built_for_another():
        _build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
