"""Build libhc.so (the CUDA library behind include/hc.h) in-tree for sm_103a.

Each .cu under csrc/ is compiled to an object in parallel with nvcc
(-gencode arch=compute_103a,code=sm_103a) and the objects are linked into
``_build/libhc.so`` with the CUDA runtime linked statically. The Python
binding's extension module (csrc/binding.cpp) is compiled beside them against
torch's headers, where torch is installed. What is newer than its sources and
headers is not built again, except a binding made for another torch or Python.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import importlib.util
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
STAMP = os.path.join(BUILD, "_hc_native.stamp")
BINDING = os.path.join(CSRC, "binding.cpp")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libhc")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newer(out: str, inputs) -> bool:
    if not os.path.exists(out):
        return False
    t = os.path.getmtime(out)
    return all(os.path.getmtime(p) <= t for p in inputs)


def _headers():
    return glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]


def torch_stamp():
    """What the binding is compiled against besides its sources: torch (its
    tensor layout is compiled in) and the interpreter. None without torch."""
    try:
        spec = importlib.util.find_spec("torch")
    except (ImportError, ValueError):  # ValueError: torch is blocked in sys.modules
        spec = None
    if spec is None or not spec.origin:
        return None
    tdir = os.path.dirname(os.path.abspath(spec.origin))
    parts = [tdir, sysconfig.get_config_var("EXT_SUFFIX")]
    for name in ("version.py", os.path.join("lib", "libtorch_python.so")):
        path = os.path.join(tdir, name)
        if os.path.exists(path):
            st = os.stat(path)
            parts.append(f"{name} {st.st_size} {st.st_mtime_ns}")
    return "\n".join(parts)


def binding_matches() -> bool:
    """Whether the built binding is one for the torch and interpreter at hand."""
    try:
        with open(STAMP) as f:
            return f.read() == torch_stamp()
    except OSError:
        return False


def _lib_up_to_date() -> bool:
    return _newer(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def _binding_up_to_date() -> bool:
    return _newer(NATIVE, [BINDING] + _headers()) and binding_matches()


def up_to_date() -> bool:
    return _lib_up_to_date() and (torch_stamp() is None or _binding_up_to_date())


def _run(cmd, what):
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{r.stdout}\n{r.stderr}")


def _build_binding(nvcc: str, objdir: str) -> None:
    """The binding's extension module (host compiler), then its stamp."""
    stamp = torch_stamp()
    import torch

    tdir = os.path.dirname(os.path.abspath(torch.__file__))
    tlib = os.path.join(tdir, "lib")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    obj = os.path.join(objdir, "binding.cpp.o")
    tmp = NATIVE + f".{os.getpid()}.tmp"
    _run(["g++", "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={abi}", "-I", INCLUDE,
          "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(tdir, "include"),
          "-isystem", os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
          "-isystem", cuda, "-c", BINDING, "-o", obj], "compiling the binding")
    _run(["g++", "-shared", "-o", tmp, obj, "-L", tlib, "-ltorch_python", "-ltorch_cpu",
          "-lc10_cuda", "-lc10", "-ldl", f"-Wl,-rpath,{tlib}"], "linking the binding")
    if os.path.exists(STAMP):
        os.remove(STAMP)  # no moment at which another module's stamp fits this one
    os.replace(tmp, NATIVE)
    tmp = STAMP + f".{os.getpid()}.tmp"
    with open(tmp, "w") as f:
        f.write(stamp)
    os.replace(tmp, STAMP)


def _build_lib(nvcc: str, objdir: str, verbose_ptxas: bool) -> None:
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2",
                    "-I", INCLUDE, "-I", CSRC]
    if verbose_ptxas or os.environ.get("HC_PTXAS_VERBOSE") == "1":
        flags += ["-Xptxas", "-v"]

    def one(src):
        obj = os.path.join(objdir, os.path.basename(src) + ".o")
        r = subprocess.run([nvcc, *flags, "-c", src, "-o", obj], capture_output=True, text=True)
        return src, obj, r

    objs, logs = [], []
    with cf.ThreadPoolExecutor(max_workers=min(12, os.cpu_count() or 4)) as ex:
        for src, obj, r in ex.map(one, sources()):
            logs.append(f"== {os.path.basename(src)}\n{r.stdout}{r.stderr}")
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
            objs.append(obj)
    with open(os.path.join(BUILD, "nvcc.log"), "w") as f:
        f.write("\n".join(logs))
    tmp = LIB + f".{os.getpid()}.tmp"
    _run([nvcc, *ARCH, "-shared", "-o", tmp, *objs], "link")
    os.replace(tmp, LIB)


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    """Builds what is out of date (everything with `force`). Without torch the
    library alone: only the binding takes torch tensors."""
    lib = force or not _lib_up_to_date()
    binding = torch_stamp() is not None and (force or not _binding_up_to_date())
    if not lib and not binding:
        return LIB
    nvcc = _nvcc()
    objdir = os.path.join(BUILD, "obj")
    os.makedirs(objdir, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=1) as ex:
        beside = ex.submit(_build_binding, nvcc, objdir) if binding else None
        if lib:
            _build_lib(nvcc, objdir, verbose_ptxas)
        if beside:
            beside.result()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose_ptxas=True))
