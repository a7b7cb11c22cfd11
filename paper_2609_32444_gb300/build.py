"""Build libcis.so (CUDA, sm_103a) in-tree with nvcc, and the native part of the
binding (C++, against the installed PyTorch) with g++.

Each .cu file compiles to an object in parallel, then nvcc links the shared
library next to this file.  Rebuilds only when a source or header is newer
than what was built.
"""

from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB_PATH = os.path.join(PKG, "libcis.so")

NATIVE_SRC = os.path.join(CSRC, "cis_native.cpp")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-std=c++17", "-O3", "-lineinfo", *ARCH, "-Xcompiler", "-fPIC,-fvisibility=hidden",
              f"-I{INCLUDE}", f"-I{CSRC}"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libcis")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(
        os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [__file__]


def native_path() -> str:
    """The binding's native module, one per Python and PyTorch version."""
    import torch
    tag = f"{sys.version_info[0]}{sys.version_info[1]}_{torch.__version__}".replace("+", "_")
    return os.path.join(PKG, f"_cis_native_{tag}.so")


def _newer(path, deps) -> bool:
    return os.path.exists(path) and all(
        os.path.getmtime(d) <= os.path.getmtime(path) for d in deps)


def up_to_date() -> bool:
    return _newer(LIB_PATH, _deps()) and _newer(
        native_path(), [NATIVE_SRC, os.path.join(INCLUDE, "cis.h"), __file__])


def _compile_native():
    import torch
    out = native_path()
    base = os.path.dirname(torch.__file__)
    libs = os.path.join(base, "lib")
    cuda = os.path.dirname(os.path.dirname(nvcc()))
    tmp = out + f".tmp{os.getpid()}"
    cmd = ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-isystem", os.path.join(base, "include"),
           "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-isystem", sysconfig.get_paths()["include"], "-isystem",
           os.path.join(cuda, "include"), f"-I{INCLUDE}", NATIVE_SRC, "-o", tmp,
           f"-L{libs}", f"-Wl,-rpath,{libs}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
           "-lc10_cuda", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed on {NATIVE_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)
    return out, r.stdout + r.stderr


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not force and up_to_date():
        return LIB_PATH
    os.makedirs(BUILD_DIR, exist_ok=True)
    cc = nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []

    def compile_one(src):
        obj = os.path.join(BUILD_DIR, os.path.basename(src) + ".o")
        cmd = [cc, *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stdout + r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(_sources()) + 1) as ex:
        native = ex.submit(_compile_native)
        results = list(ex.map(compile_one, _sources()))
        native.result()
    if verbose or ptxas_info:
        for _, log in results:
            if log.strip():
                print(log)
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [cc, "-shared", *ARCH, "-o", tmp, *[o for o, _ in results]]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
