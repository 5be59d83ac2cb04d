"""In-tree build: libpolarquant.so with nvcc for sm_100a (cross-compiles without a GPU), and the extension module
_pq_binding.so that calls it from PyTorch tensors."""
from __future__ import annotations

import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpolarquant.so")
BINDING = os.path.join(HERE, "_pq_binding.so")
SOURCES = ["pq_host.cu", "pq_encode.cu", "pq_decode.cu", "pq_general.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared", "--threads", "0"]
HEADER = os.path.join(HERE, "..", "include", "polarquant.h")


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def _stale(target, deps):
    return not os.path.exists(target) or os.path.getmtime(target) < _newest(deps)


def _run(cmd, what, verbose):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(what + " failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    deps = srcs + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))] + [HEADER]
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if force or _stale(LIB, deps):
        _run([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + srcs, "nvcc", verbose)
    build_binding(force, verbose)
    return LIB


def build_binding(force: bool = False, verbose: bool = False) -> str:
    src = os.path.join(CSRC, "pq_binding.cpp")
    if force or _stale(BINDING, [src, HEADER]):
        import torch
        from torch.utils import cpp_extension
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
        includes = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], cuda]
        torch_lib = os.path.join(os.path.dirname(torch.__file__), "lib")
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wno-attributes",
               "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
        cmd += ["-isystem" + p for p in includes] + ["-o", BINDING, src]
        # the torch libraries are loaded by `import torch`; the library lies beside the module
        cmd += ["-L" + torch_lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-L" + HERE, "-l:libpolarquant.so",
                "-Wl,-rpath,$ORIGIN"]
        _run(cmd, "g++", verbose)
    return BINDING


if __name__ == "__main__":
    print(build(force=True, verbose=True))
