"""Builds libspade.so (the C-ABI library) in-tree with nvcc for sm_103a, and its Python binding.

Each .cu under csrc/ is compiled to an object in parallel, then linked into
``paper_2608_13076_gb300/lib/libspade.so`` with the CUDA runtime linked
statically; csrc/binding.cpp becomes ``lib/_spade_native.so``, an extension
module over the installed torch.  A rebuild happens only when a source is newer
than the outputs, or the torch or Python that the module was built for is not the
one at hand.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
BUILD_DIR = os.path.join(HERE, "_build")
LIB_DIR = os.path.join(HERE, "lib")
LIB_PATH = os.path.join(LIB_DIR, "libspade.so")
NATIVE_PATH = os.path.join(LIB_DIR, "_spade_native.so")
STAMP_PATH = os.path.join(LIB_DIR, "_spade_native.stamp")  # what the extension module was built for
BINDING = os.path.join(CSRC, "binding.cpp")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE]


def _nvcc():
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the SPADE library needs the CUDA 13 toolkit")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + [BINDING] + sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))) \
        + [os.path.join(INCLUDE, "spade.h"), os.path.abspath(__file__)]


def _built_for() -> str:
    import torch
    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def up_to_date() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH) or not os.path.exists(STAMP_PATH):
        return False
    with open(STAMP_PATH) as f:
        if f.read() != _built_for():
            return False
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    return all(os.path.getmtime(d) <= t for d in _deps())


def _run(cmd, what):
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{r.stdout}\n{r.stderr}")
    return r


def _compile_binding(cuda_home):
    """csrc/binding.cpp -> object, against the installed torch and Python headers."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    obj = os.path.join(BUILD_DIR, "binding.o")
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-c", BINDING, "-o", obj,
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", INCLUDE, "-isystem", inc,
          "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
          "-isystem", os.path.join(cuda_home, "include"), "-isystem", sysconfig.get_paths()["include"]],
         "g++ on binding.cpp")
    return obj


def _link_binding(obj):
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE_PATH + ".tmp"
    _run([os.environ.get("CXX", "g++"), "-shared", "-o", tmp, obj, LIB_PATH, "-L", lib, "-lc10", "-lc10_cuda",
          "-ltorch_cpu", "-ltorch_python", f"-Wl,-rpath,$ORIGIN,-rpath,{lib}"], "link of the Python binding")
    os.replace(tmp, NATIVE_PATH)
    with open(STAMP_PATH, "w") as f:
        f.write(_built_for())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source for sm_103a and link libspade.so; returns its path."""
    if not force and up_to_date():
        return LIB_PATH
    nvcc = _nvcc()
    os.makedirs(BUILD_DIR, exist_ok=True)
    os.makedirs(LIB_DIR, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(BUILD_DIR, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc] + NVCC_FLAGS + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {os.path.basename(src)}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr)
        return obj

    cuda_home = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    with ThreadPoolExecutor(max_workers=max(1, min(16, os.cpu_count() or 1))) as ex:
        binding = ex.submit(_compile_binding, cuda_home)
        objs = list(ex.map(compile_one, sources()))
        binding_obj = binding.result()
    tmp = LIB_PATH + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-Xlinker", "-soname=libspade.so", "-o", tmp] + objs + ["-lcudart_static", "-ldl", "-lpthread", "-lrt"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PATH)
    _link_binding(binding_obj)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
