"""Builds liblla.so (the CUDA library behind include/lla.h) in-tree for sm_103a, and _lla_native.so
(csrc/lla_binding.cpp: the native marshalling of the Python binding, linked to liblla.so beside it).

Each translation unit is compiled by nvcc in parallel, then linked into
paper_2607_15456_gb300/liblla.so with the CUDA runtime linked statically, so the library
needs nothing but the driver at run time.  The binding is one host translation unit against torch's
headers, compiled beside them; where it cannot be built, calls are marshalled in Python.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "liblla.so")
NATIVE = os.path.join(PKG, "_lla_native.so")
BINDING = os.path.join(CSRC, "lla_binding.cpp")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
         "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newer(target: str, deps) -> bool:
    return os.path.exists(target) and all(os.path.getmtime(p) <= os.path.getmtime(target) for p in deps)


def library_up_to_date() -> bool:
    return _newer(LIB, _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) +
                  [os.path.join(ROOT, "include", "lla.h"), __file__])


def binding_abi() -> str:
    """What _lla_native.so is compiled against: the interpreter's and torch's C++ ABI."""
    import torch
    return f"{sysconfig.get_config_var('SOABI')} torch {torch.__version__}"


def binding_up_to_date() -> bool:
    try:
        with open(NATIVE + ".abi") as f:
            abi = f.read()
    except OSError:
        return False
    return abi == binding_abi() and _newer(NATIVE, [BINDING, os.path.join(ROOT, "include", "lla.h"), __file__])


def _run(cmd, what: str):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{what} failed:\n{res.stdout}\n{res.stderr}")


def compile_binding() -> str:
    """lla_binding.cpp as an object file, against this interpreter's Python and torch headers."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")
    obj = os.path.join(BUILD, "lla_binding.o")
    _run(["g++", "-O2", "-std=c++17", "-fPIC", "-Wall", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          "-I" + os.path.join(ROOT, "include"), "-I" + sysconfig.get_paths()["include"], "-isystem", inc,
          "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", cuda, "-c", BINDING, "-o", obj],
         "g++ on lla_binding.cpp")
    return obj


def link_binding(obj: str) -> None:
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".tmp%d" % os.getpid()
    _run(["g++", "-shared", obj, "-o", tmp, "-L" + PKG, "-l:liblla.so", "-Wl,-rpath,$ORIGIN", "-L" + lib, "-ltorch_python",
          "-ltorch_cpu", "-lc10", "-lc10_cuda"], "linking _lla_native.so")
    if os.path.exists(NATIVE + ".abi"):
        os.remove(NATIVE + ".abi")  # never a new note beside an old module
    os.replace(tmp, NATIVE)
    with open(NATIVE + ".abi", "w") as f:
        f.write(binding_abi())


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    """Compiles every csrc/*.cu for sm_103a and links liblla.so, and builds the binding's native
    marshalling beside it; returns the library's path."""
    library, binding = force or not library_up_to_date(), force or not binding_up_to_date()
    if not library and not binding:
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        cmd = [nvcc, *ARCH, *FLAGS, "-c", src, "-o", obj]
        if ptxas_info:
            cmd.insert(1, "-Xptxas=-v")
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
        if verbose or ptxas_info:
            sys.stderr.write(res.stdout + res.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 2)) as ex:
        obj = ex.submit(compile_binding) if binding else None
        objs = list(ex.map(compile_one, _sources())) if library else []
    if library:
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", *objs, "-o", tmp]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")
        os.replace(tmp, LIB)
    if binding:
        try:
            link_binding(obj.result())
        except (RuntimeError, OSError, ImportError) as e:  # no g++, no headers, another torch
            if os.path.exists(NATIVE):
                os.remove(NATIVE)  # of an older source
            sys.stderr.write(f"_lla_native.so was not built, calls will be marshalled in Python: {e}\n")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv,
                ptxas_info="--ptxas-info" in sys.argv))
