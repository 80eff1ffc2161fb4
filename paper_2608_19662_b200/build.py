"""Builds librecache.so (nvcc for sm_100a, cross-compiles without a GPU) and the Python entry points
_native.so (g++ against torch) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librecache.so")
NATIVE = os.path.join(HERE, "_native.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = (os.environ.get("RECACHE_NVCC_EXTRA", "").split()) + ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


def headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def stale() -> bool:
    return _older(LIB, sources() + headers()) or _older(NATIVE, [os.path.join(CSRC, "native.cpp")] + headers())


def native_command():
    import torch
    from torch.utils import cpp_extension
    lib_dir = os.path.join(os.path.dirname(torch.__file__), "lib")
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include"),
                                           os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    return (["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
             "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi()] + ["-I" + p for p in inc] +
            [os.path.join(CSRC, "native.cpp"), "-o", NATIVE, "-L" + lib_dir, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
             "-lc10_cuda"])


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not stale():
        return LIB
    objs = []
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    native = subprocess.Popen(native_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    procs = []
    for src in sources():
        obj = os.path.join(HERE, "build", os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj] + (["-Xptxas", "-v"] if verbose else [])
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
    cmd = [NVCC, "-shared", "-o", LIB, *objs, "-lcudart"]
    subprocess.check_call(cmd)
    out, _ = native.communicate()
    if native.returncode:
        sys.stderr.write(out)
        raise RuntimeError("g++ failed on native.cpp")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
