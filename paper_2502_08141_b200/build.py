"""Compile the CUDA sources into ``liblowra.so`` next to this file (sm_100a only), and the Python binding's native part into a
``_py_calls.*.so`` whose name says for which Python and torch."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

from . import PY_CALLS_PATH as PY_CALLS

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblowra.so")
PY_CALLS_SOURCE = os.path.join(CSRC, "py_calls.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--ftz=false", "--prec-div=true", "--prec-sqrt=true", "--fmad=true",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "-Xptxas", "-v",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(PY_CALLS):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(PY_CALLS))
    deps = sources() + [PY_CALLS_SOURCE] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _py_calls_command():
    import sysconfig

    import torch
    from torch.utils import cpp_extension

    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    includes = [ROOT + "/include", sysconfig.get_paths()["include"], *cpp_extension.include_paths(device_type="cuda")]
    return [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-w", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            "-DTORCH_API_INCLUDE_EXTENSION_H", *("-I" + i for i in includes), PY_CALLS_SOURCE, "-o", PY_CALLS, "-L" + libs, "-Wl,-rpath," + libs,
            "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    """nvcc -> liblowra.so.  Cross-compiles without a GPU."""
    if not force and not _stale():
        return LIB
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    run = lambda cmd: subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)  # noqa: E731
    py_calls = run(_py_calls_command())
    objs = []
    procs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        procs.append((src, run([nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj])))

    def finished(src, p) -> bool:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        return p.returncode == 0

    done = [finished(src, p) for src, p in procs]
    if all(done):
        subprocess.run([nvcc, "-shared", "-o", LIB, *objs, "-lcudart"], check=True)
    # (last: where it does not compile, the library is there all the same, and the calls take the interpreted way)
    if not finished(PY_CALLS_SOURCE, py_calls) or not all(done):
        raise RuntimeError("compilation failed")
    return LIB


if __name__ == "__main__":
    build(force=True, verbose=True)
    print(LIB)
