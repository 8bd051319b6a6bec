"""Builds the CUDA library (nvcc, sm_100a only) and the extension module that binds it (g++), in-tree.

    python -m paper_2604_09244_b200.build
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libmvla_prune.so")
EXT = os.path.join(PKG, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["api.cu", "salience.cu", "fused.cu", "stream.cu", "select.cu", "compact.cu", "step.cu", "patch.cu", "patch_step.cu", "salience_noalloc.cu"]
BINDING = "binding.cpp"
HEADER = os.path.join(ROOT, "include", "mvla_prune.h")


def _newer(target: str, deps) -> bool:
    return os.path.exists(target) and all(os.path.getmtime(d) <= os.path.getmtime(target) for d in deps)


def _stale() -> bool:
    cuda = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != BINDING] + [HEADER]
    return not (_newer(LIB, cuda) and _newer(EXT, [os.path.join(CSRC, BINDING), HEADER]))


def _compile_cuda(tmp: str, verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC",
             "-I", os.path.join(ROOT, "include"), "-I", CSRC] + (["-Xptxas=-v"] if verbose else [])
    flags += os.environ.get("MVLA_NVCC_FLAGS", "").split()     # extra compiler flags

    def one(f):
        obj = os.path.join(tmp, f + ".o")
        subprocess.run([nvcc, *flags, "-c", os.path.join(CSRC, f), "-o", obj], check=True)
        return obj
    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
        objs = list(pool.map(one, SOURCES))
    subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs, "-lcudart"], check=True)


def _compile_binding() -> None:
    import torch
    from torch.utils import cpp_extension
    inc = cpp_extension.include_paths() + [os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include",
                                           sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for d in inc:
        cmd += ["-isystem", d]
    # torch's own libraries are loaded with `import torch`; the CUDA library lies beside the module
    cmd += [os.path.join(CSRC, BINDING), "-o", EXT, "-L", libs, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
            "-lc10_cuda", "-L", PKG, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    with tempfile.TemporaryDirectory() as tmp:
        _compile_cuda(tmp, verbose)
    _compile_binding()
    return LIB


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
