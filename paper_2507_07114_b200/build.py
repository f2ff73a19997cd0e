"""Build the CUDA library in-tree with nvcc for sm_100a, and the binding's marshalling module (no JIT cache)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "liblossy_b200.so")
CHECK_LIB_PATH = os.path.join(PKG_DIR, "liblossy_b200_check.so")   # the debug build: -DLOSSY_DEVCHECK (index checks in the kernels)
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")
SOURCES = ["lossy_api.cu", "lossy_noalloc.cu"]
HEADERS = ["lossy_divide.h", "lossy_device.cuh", "lossy_kernels.cuh", "lossy_tma.cuh", "lossy_gather.cuh", "lossy_phase_tma.cuh", "lossy_register.cuh", "lossy_diag.cuh", os.path.join("..", "..", "include", "lossy.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-fmad=false",                      # every fp32 operation of the contract is rounded on its own
    "-Xcompiler", "-fPIC", "-shared",
]


def marshal_path() -> str:
    """The binding's marshalling module. It uses the C++ interfaces of one Python and one torch, which its name holds: with others another
    file is wanted, missing until it is built."""
    import torch

    return os.path.join(PKG_DIR, f"_marshal-{sysconfig.get_config_var('SOABI')}-torch-{torch.__version__}.so")


def _stale(lib: str) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = ([MARSHAL_SOURCE] if os.path.basename(lib).startswith("_marshal") else [os.path.join(CSRC, s) for s in SOURCES + HEADERS]) + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def _marshal_command(out: str) -> list:
    """g++ on marshal.cpp, against the headers of the Python and the torch that run this."""
    import torch

    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
            *["-isystem" + d for d in include], MARSHAL_SOURCE, "-o", out, "-L" + os.path.join(root, "lib"),
            "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile liblossy_b200.so, its debug twin liblossy_b200_check.so and the binding's marshalling module next to this file
    (the compilers side by side); returns the path of the normal library."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    jobs = []
    marshal = marshal_path()
    if force or _stale(marshal):
        jobs.append((marshal, subprocess.Popen(_marshal_command(marshal + ".tmp"), stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)))
    for lib, extra in ((LIB_PATH, []), (CHECK_LIB_PATH, ["-DLOSSY_DEVCHECK=1"])):
        if not force and not _stale(lib):
            continue
        cmd = [nvcc, *NVCC_FLAGS, *extra, *(["-Xptxas", "-v"] if verbose and not extra else []), "-o", lib + ".tmp",
               *[os.path.join(CSRC, s) for s in SOURCES]]
        jobs.append((lib, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)))
    failed = []
    for lib, proc in jobs:
        out, err = proc.communicate()
        if verbose:
            sys.stderr.write(err)
        if proc.returncode != 0:
            failed.append(os.path.basename(lib) + ":\n" + out + err)
        else:
            os.replace(lib + ".tmp", lib)
    if failed:
        raise RuntimeError("build failed:\n" + "\n".join(failed))
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
