"""Builds libobcache.so (the C-ABI CUDA library, nvcc for sm_100a) and _native.so (its binding for torch tensors, g++) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libobcache.so")
NATIVE = os.path.join(PKG, "_native.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def native_command() -> list[str]:
    """g++ command of the binding: torch's headers and libraries, the C ABI, Python's headers."""
    from torch.utils import cpp_extension
    inc = [a for d in cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
           for a in ("-isystem" if "torch" in d else "-I", d)]
    libs = [f"-L{d}" for d in cpp_extension.library_paths("cuda")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", *inc, os.path.join(CSRC, "binding.cpp"), "-o", NATIVE, *libs,
            "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10", f"-L{PKG}", "-l:libobcache.so", "-Wl,-rpath,$ORIGIN"]


def stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cpp")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library (cross-compiles without a GPU)."""
    if not force and not stale():
        return LIB
    objs = []
    procs = []
    bdir = os.path.join(PKG, "_build")
    os.makedirs(bdir, exist_ok=True)
    for src in sources():
        obj = os.path.join(bdir, os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj] + (["-Xptxas", "-v"] if verbose else [])
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.check_call([NVCC, "-shared", "-o", LIB, *objs])  # static cudart (nvcc default)
    subprocess.check_call(native_command())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
