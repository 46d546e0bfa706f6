"""Build libchunkkv.so (CUDA, sm_100a) with nvcc and the binding's native part with g++, in-tree.

Usage: ``python -m paper_2502_00299_b200.build [--force]``. Objects go to ``_build/`` inside the
package; the shared library is written next to this file so that it ships with the package.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
BUILD_DIR = os.path.join(PKG_DIR, "_build")
LIB_PATH = os.path.join(PKG_DIR, "libchunkkv.so")
INCLUDE_DIR = os.path.join(os.path.dirname(PKG_DIR), "include")
SOURCES = ("api.cu", "score.cu", "layer_resident.cu", "model_kernel.cu", "token_kernel.cu", "select.cu", "select_cluster.cu", "gather.cu", "diagnostics.cu", "score_noalloc.cu")
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
]


def native_path() -> str:
    """The extension module used by binding.py. Its name holds the versions of torch and Python that it was built for and that run now."""
    import torch
    return os.path.join(PKG_DIR, f"_native-torch{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; libchunkkv needs the CUDA toolkit to build")
    return cand


def _deps_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    paths += [os.path.join(INCLUDE_DIR, f) for f in os.listdir(INCLUDE_DIR)] + [os.path.abspath(__file__)]
    return max(os.path.getmtime(p) for p in paths)


def is_current() -> bool:
    return all(os.path.exists(p) and os.path.getmtime(p) >= _deps_mtime() for p in (LIB_PATH, native_path()))


def _compile_native() -> str:
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    obj = os.path.join(BUILD_DIR, "native.o")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(root, "include"),
           "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
           "-c", os.path.join(CSRC, "native.cpp"), "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"g++ failed on native.cpp:\n{res.stdout}\n{res.stderr}")
    return obj


def _link_native(obj: str) -> None:
    import torch
    lib = os.path.join(os.path.dirname(os.path.abspath(torch.__file__)), "lib")
    for f in os.listdir(PKG_DIR):                      # of other versions
        if f.startswith("_native") and f.endswith(".so"):
            os.remove(os.path.join(PKG_DIR, f))
    cmd = ["g++", "-shared", "-o", native_path(), obj, "-L", PKG_DIR, "-l:libchunkkv.so", "-Wl,-rpath,$ORIGIN", "-L", lib, "-ltorch_python", "-ltorch",
           "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link of {native_path()} failed:\n{res.stdout}\n{res.stderr}")


def report_path(src: str) -> str:
    """What ptxas said of a source file's kernels (registers, spills, shared memory)."""
    return os.path.join(BUILD_DIR, src.replace(".cu", ".ptxas.txt"))


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(BUILD_DIR, src.replace(".cu", ".o"))
    cmd = [_nvcc(), *NVCC_FLAGS, "-Xptxas", "-v", "-I", INCLUDE_DIR, "-c", os.path.join(CSRC, src), "-o", obj]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
    with open(report_path(src), "w") as f:
        f.write(res.stderr)
    if verbose:
        sys.stderr.write(res.stderr)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_100a and link the shared library and the extension module. Returns the library's path."""
    if not force and not verbose and is_current():
        return LIB_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as pool:
        native = pool.submit(_compile_native)
        objs = list(pool.map(lambda s: _compile(s, verbose), SOURCES))
    cmd = [_nvcc(), "-Wno-deprecated-gpu-targets", "-shared", "-o", LIB_PATH, *objs, "-lcudart"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
    _link_native(native.result())
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
