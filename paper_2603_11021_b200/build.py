"""Compile the CUDA library in-tree for sm_100a with nvcc."""
from __future__ import annotations

import glob
import os
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
LIB = os.path.join(PKG, "libllvq.so")
NATIVE = os.path.join(PKG, "_native.so")            # the Python module that calls it on PyTorch tensors (csrc/binding.cpp)
BINDING = os.path.join(PKG, "csrc", "binding.cpp")

NVCC_FLAGS = [
    "-O3", "-std=c++17",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-lineinfo",
    "-Xcompiler", "-fPIC",
]
OBJ_DIR = os.path.join(PKG, "build")


def sources() -> list[str]:
    src = sorted(glob.glob(os.path.join(PKG, "csrc", "*.cu")) + glob.glob(os.path.join(PKG, "csrc", "*.cpp")))
    return [f for f in src if f != BINDING]


def _headers() -> list[str]:
    return glob.glob(os.path.join(ROOT, "include", "*.h"))


def _inputs() -> list[str]:
    return sources() + _headers() + glob.glob(os.path.join(PKG, "csrc", "*.h")) + glob.glob(os.path.join(PKG, "csrc", "*.cuh"))


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _inputs())


def build(force: bool = False, verbose: bool = False) -> str:
    """Build libllvq.so and _native.so next to this file; returns the library's path."""
    if force or is_stale():
        _build_library(verbose)
    if force or native_is_stale():
        _build_native()
    return LIB


def native_stamp() -> str:
    """What _native.so is compiled against beside its sources: it holds inline code of PyTorch's and Python's headers."""
    import sys
    import torch
    return f"built for torch {torch.__version__}, cxx11 {int(torch.compiled_with_cxx11_abi())}, python {sys.version_info.major}.{sys.version_info.minor}"


def native_matches() -> bool:
    """Whether _native.so, which carries its stamp, was built for the PyTorch and Python that run."""
    with open(NATIVE, "rb") as f:
        return native_stamp().encode() + b"\0" in f.read()


def native_is_stale() -> bool:
    if not os.path.exists(NATIVE) or not native_matches():
        return True
    return any(os.path.getmtime(NATIVE) < os.path.getmtime(f) for f in [BINDING] + _headers())


def _build_native() -> None:
    """The Python module: plain C++ against PyTorch's headers, linked to libllvq.so beside it."""
    import sysconfig
    import torch
    root = os.path.join(os.path.dirname(torch.__file__))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = NATIVE + f".{os.getpid()}.tmp"
    subprocess.check_call([
        os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
        f'-DLLVQ_BUILT_FOR="{native_stamp()}"',
        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(root, "include"), "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
        "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], BINDING, "-o", tmp, "-L", PKG, "-lllvq",
        "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, NATIVE)


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, os.path.splitext(os.path.basename(src))[0] + f".{os.getpid()}.o")
        subprocess.check_call([nvcc, *NVCC_FLAGS, *extra, "-I", os.path.join(ROOT, "include"), "-c", src, "-o", obj])
        return obj

    # one nvcc process per translation unit, side by side
    from concurrent.futures import ThreadPoolExecutor
    with ThreadPoolExecutor(max_workers=min(8, len(sources()))) as ex:
        objs = list(ex.map(compile_one, sources()))
    tmp = LIB + f".{os.getpid()}.tmp"
    subprocess.check_call([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs])
    os.replace(tmp, LIB)
    for o in objs:
        os.remove(o)


if __name__ == "__main__":
    print(build(force=True, verbose=True))
