"""Build libgbs.so (the C-ABI CUDA library, nvcc for sm_100a) and _native.so (the binding's native call path) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgbs.so")
NATIVE = os.path.join(PKG, "_native.so")
NATIVE_SRC = os.path.join(CSRC, "gbs_torch.cpp")

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")        # its toolkit's headers serve _native.so as well
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC,-Wall",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = sources() + [NATIVE_SRC] + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def native_command(obj: str) -> list:
    """g++ command that compiles the native call path against this interpreter's torch."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    return ["g++", "-O3", "-std=c++20", "-fPIC", "-Wall", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            "-I", os.path.join(ROOT, "include"), "-isystem", inc,
            "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", sysconfig.get_paths()["include"],
            "-isystem", os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), "-c", NATIVE_SRC, "-o", obj]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libgbs.so; returns its path."""
    if not force and not is_stale():
        return LIB
    objs = []
    build_dir = os.path.join(PKG, "_build")
    os.makedirs(build_dir, exist_ok=True)
    procs = []
    headers = max(os.path.getmtime(f) for pat in (os.path.join(CSRC, "*.h"), os.path.join(CSRC, "*.cuh"),
                                                  os.path.join(ROOT, "include", "*.h"), __file__) for f in glob.glob(pat))

    def fresh(obj, src):
        return not force and not verbose and os.path.exists(obj) and os.path.getmtime(obj) > max(headers, os.path.getmtime(src))

    for src in sources():
        obj = os.path.join(build_dir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if fresh(obj, src):
            continue
        cmd = [NVCC] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        procs.append((cmd, subprocess.Popen(cmd)))
    native_obj = os.path.join(build_dir, "gbs_torch.o")
    if not fresh(native_obj, NATIVE_SRC):
        cmd = native_command(native_obj)
        procs.append((cmd, subprocess.Popen(cmd)))
    for cmd, pr in procs:
        if pr.wait() != 0:
            raise RuntimeError("compilation failed: " + " ".join(cmd))
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([NVCC, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    # libgbs.so is found beside _native.so; torch's libraries are already loaded when the package is imported
    import torch
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    subprocess.check_call(["g++", "-shared", "-o", tmp, native_obj, "-L", PKG, "-lgbs", "-Wl,-rpath,$ORIGIN", "-L", tlib,
                           "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    os.replace(tmp, NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
