"""Build libhc.so (the CUDA library behind include/hc.h) in-tree for sm_103a.

Each .cu under csrc/ is compiled to an object in parallel with nvcc
(-gencode arch=compute_103a,code=sm_103a) and the objects are linked into
``_build/libhc.so`` with the CUDA runtime linked statically. The Python
binding's extension module (csrc/binding.cpp) is compiled beside them against
torch's headers. A build is skipped when both are newer than
every source and header.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "libhc.so")
NATIVE = os.path.join(BUILD, "_hc_native.so")
BINDING = os.path.join(CSRC, "binding.cpp")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libhc")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _inputs():
    return sources() + [BINDING] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]


def up_to_date() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return False
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    return all(os.path.getmtime(p) <= t for p in _inputs())


def _native_commands(nvcc: str, obj: str, out: str):
    """The binding's compile and link commands (host compiler)."""
    import torch

    tdir = os.path.dirname(os.path.abspath(torch.__file__))
    tlib = os.path.join(tdir, "lib")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    comp = ["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={abi}", "-I", INCLUDE,
            "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(tdir, "include"),
            "-isystem", os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
            "-isystem", cuda, "-c", BINDING, "-o", obj]
    link = ["g++", "-shared", "-o", out, obj, "-L", tlib, "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", "-ldl", f"-Wl,-rpath,{tlib}"]
    return comp, link


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    nvcc = _nvcc()
    objdir = os.path.join(BUILD, "obj")
    os.makedirs(objdir, exist_ok=True)
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2",
                    "-I", INCLUDE, "-I", CSRC]
    if verbose_ptxas or os.environ.get("HC_PTXAS_VERBOSE") == "1":
        flags += ["-Xptxas", "-v"]

    def one(src):
        obj = os.path.join(objdir, os.path.basename(src) + ".o")
        r = subprocess.run([nvcc, *flags, "-c", src, "-o", obj], capture_output=True, text=True)
        return src, obj, r

    native_obj = os.path.join(objdir, "binding.cpp.o")
    native_tmp = NATIVE + f".{os.getpid()}.tmp"
    native_comp, native_link = _native_commands(nvcc, native_obj, native_tmp)

    def run(cmd, what):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"{what} failed:\n{r.stdout}\n{r.stderr}")

    objs, logs = [], []
    with cf.ThreadPoolExecutor(max_workers=min(12, os.cpu_count() or 4)) as ex:
        native = ex.submit(run, native_comp, "compiling the binding")
        for src, obj, r in ex.map(one, sources()):
            logs.append(f"== {os.path.basename(src)}\n{r.stdout}{r.stderr}")
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
            objs.append(obj)
        native.result()
    with open(os.path.join(BUILD, "nvcc.log"), "w") as f:
        f.write("\n".join(logs))
    tmp = LIB + f".{os.getpid()}.tmp"
    r = subprocess.run([nvcc, *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    run(native_link, "linking the binding")
    os.replace(native_tmp, NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose_ptxas=True))
