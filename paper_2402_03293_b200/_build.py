"""In-tree build of the CUDA library (nvcc, sm_100a only)."""
from __future__ import annotations

import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libflora.so")
NATIVE_SOURCE = "flora_py.cpp"
SOURCES = ["flora_api.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared", "--fmad=false", "-Xptxas", "-v"]


def _newest_source_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != NATIVE_SOURCE]
    paths.append(os.path.join(os.path.dirname(HERE), "include", "flora.h"))
    return max(os.path.getmtime(p) for p in paths)


def native_path() -> str:
    """The Python side of binding.py (argument marshalling).  It reads torch's C++ objects, whose layout belongs to one build of torch
    and Python: the name says for which it was made, so another one does not load it."""
    import torch
    return os.path.join(HERE, f"_native-{sysconfig.get_config_var('SOABI')}-torch{torch.__version__}.so")


def build_native(force: bool = False) -> str:
    """Compile csrc/flora_py.cpp (g++ only; needs libflora.so, which it calls) where missing or stale."""
    native = native_path()
    src = os.path.join(CSRC, NATIVE_SOURCE)
    newest = max(os.path.getmtime(src), os.path.getmtime(os.path.join(os.path.dirname(HERE), "include", "flora.h")))
    if not force and os.path.exists(native) and os.path.getmtime(native) >= newest:
        return native
    import torch
    root = os.path.dirname(torch.__file__)
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f"-I{root}/include", f"-I{root}/include/torch/csrc/api/include", "-I/usr/local/cuda/include",
           f"-I{sysconfig.get_paths()['include']}", src, "-o", native + ".tmp", f"-L{root}/lib", "-ltorch_python", "-ltorch_cpu", "-lc10",
           "-lc10_cuda", f"-L{HERE}", "-l:libflora.so", "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode:
        print(res.stderr)
        raise RuntimeError("g++ failed building the native side of binding.py")
    os.replace(native + ".tmp", native)
    return native


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into paper_2402_03293_b200/libflora.so, and the Python side, where missing or stale."""
    lib = build_library(force, verbose)
    build_native(force)
    return lib


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc] + NVCC_FLAGS + [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB + ".tmp"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode:
        print(res.stdout)
        print(res.stderr)
    if res.returncode:
        raise RuntimeError("nvcc failed building libflora.so")
    with open(os.path.join(HERE, "ptxas_report.txt"), "w") as f:
        f.write(res.stderr)
    os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
