"""In-tree build of the CUDA library (nvcc, sm_100a only) and of the extension that marshals its arguments (g++ against
torch's headers).  `python -m paper_2603_15965_b200.build`."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libmolora.so")
MARSHAL_PATH = os.path.join(PKG_DIR, "_marshal.so")
MARSHAL_ABI_PATH = os.path.join(PKG_DIR, "_marshal.abi")      # what the extension was built for, written beside it

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--threads", "0", "-I", os.path.join(ROOT, "include")]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def marshal_abi() -> str:
    """The interpreter and the torch whose C++ interfaces the extension is compiled against."""
    import torch
    return f"{sys.implementation.cache_tag} torch {torch.__version__} cxx11abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)}"


def marshal_built_for() -> str:
    """What marshal_abi() was when the extension was built; empty if that is not known."""
    if not os.path.exists(MARSHAL_ABI_PATH):
        return ""
    with open(MARSHAL_ABI_PATH) as f:
        return f.read().strip()


def build_marshal(force: bool = False) -> str:
    """Compile csrc/marshal.cpp into _marshal.so beside the library it links to (no GPU, no nvcc)."""
    src = os.path.join(CSRC, "marshal.cpp")
    deps = [src] + glob.glob(os.path.join(ROOT, "include", "*.h"))
    if (not force and os.path.exists(MARSHAL_PATH) and marshal_built_for() == marshal_abi()
            and all(os.path.getmtime(p) <= os.path.getmtime(MARSHAL_PATH) for p in deps)):
        return MARSHAL_PATH
    import torch
    torch_dir = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = MARSHAL_PATH + f".{os.getpid()}.tmp"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(torch_dir, "include"),
           "-isystem", os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"), src, "-o", tmp,
           "-L", os.path.join(torch_dir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-L", PKG_DIR, "-l:libmolora.so",
           "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, MARSHAL_PATH)
    with open(MARSHAL_ABI_PATH, "w") as f:
        f.write(marshal_abi() + "\n")
    return MARSHAL_PATH


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libmolora.so next to this file (cross-compiles without a GPU)."""
    if not force and not _stale():
        build_marshal()
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB_PATH + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-shared", "-o", tmp] + sources()
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stderr)
    os.replace(tmp, LIB_PATH)
    build_marshal(force)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
