"""Builds libglide.so in-tree with nvcc for sm_103a (GB300).

Each translation unit under csrc/ is compiled in parallel into _build/, then
linked into paper_2402_02082_gb300/libglide.so (CUDA runtime linked
statically, so the library loads on a machine without a GPU too).  The Python
binding's argument marshalling (csrc/pycall.cpp) is compiled beside them
against the installed torch and linked to the library; its file carries
torch's version, whose C++ interface it uses.  A rebuild happens only when a
source or header is newer than what was built.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libglide.so")
INCLUDE = os.path.join(ROOT, "include")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "--expt-relaxed-constexpr"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    return "nvcc"


def call_module() -> str:
    """Path of the marshalling module for the installed torch."""
    import torch
    return os.path.join(PKG, f"_glidecall-{torch.__version__.replace('+', '-')}.so")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(CSRC, "*.cpp")) + glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]


def up_to_date() -> bool:
    built = (LIB, call_module())
    if not all(os.path.exists(p) for p in built):
        return False
    t = min(os.path.getmtime(p) for p in built)
    return all(os.path.getmtime(p) <= t for p in _deps())


def _compile(src: str, verbose_ptxas: bool) -> str:
    obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
    cmd = [nvcc(), *ARCH, *FLAGS, "-c", src, "-o", obj]
    if verbose_ptxas:
        cmd += ["-Xptxas", "-v"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    if verbose_ptxas:
        sys.stderr.write(r.stderr)
    return obj


def _compile_call_module() -> str:
    import torch
    at = os.path.dirname(torch.__file__)
    include = [os.path.join(at, "include"), os.path.join(at, "include", "torch", "csrc", "api", "include"),
               os.path.join(os.path.dirname(os.path.dirname(nvcc())) or "/usr/local/cuda", "include"),
               sysconfig.get_paths()["include"], INCLUDE]
    obj = os.path.join(BUILD, "pycall.o")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *(f"-I{p}" for p in include), "-c", os.path.join(CSRC, "pycall.cpp"), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"compiling pycall.cpp failed:\n{r.stdout}\n{r.stderr}")
    return obj


def _link_call_module(obj: str) -> None:
    import torch
    path = call_module()
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = [os.environ.get("CXX", "g++"), "-shared", "-o", path + ".tmp", obj, f"-L{libs}", "-ltorch_python",
           "-ltorch_cpu", "-lc10", "-lc10_cuda", f"-L{PKG}", "-lglide", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"linking the call module failed:\n{r.stdout}\n{r.stderr}")
    os.replace(path + ".tmp", path)


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    """Compile and link libglide.so and the call module; returns the library's path."""
    verbose_ptxas = verbose_ptxas or os.environ.get("GLIDE_PTXAS_VERBOSE") == "1"
    if not force and not verbose_ptxas and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    srcs = _sources()
    with concurrent.futures.ThreadPoolExecutor(max_workers=max(1, min(len(srcs) + 1, os.cpu_count() or 1))) as ex:
        call_obj = ex.submit(_compile_call_module)
        objs = list(ex.map(lambda s: _compile(s, verbose_ptxas), srcs))
    tmp = LIB + ".tmp"
    r = subprocess.run([nvcc(), *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    _link_call_module(call_obj.result())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv))
