"""Builds libmadakv.so (the C-ABI CUDA library, nvcc for sm_100a) and _native.so (its Python entry points, g++) in-tree."""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libmadakv.so")
NATIVE_SRC = os.path.join(HERE, "csrc", "py_binding.cpp")
NATIVE = os.path.join(HERE, "_native.so")
PROBE_SRC = os.path.join(HERE, "csrc", "probe", "exp2_roof.cu")
PROBE = os.path.join(HERE, "exp2_roof.bin")  # measures the exp2 roof (see the source); used by bench.py


def sources():
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def needs_build():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(HERE, "csrc", "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def build_probe(force=False):
    """The stand-alone exp2-roof probe (a small CUDA program, not part of the library)."""
    if force or not os.path.exists(PROBE) or os.path.getmtime(PROBE) < os.path.getmtime(PROBE_SRC):
        subprocess.check_call(["nvcc", "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
                               "-o", PROBE, PROBE_SRC])
    return PROBE


def build_native(force=False):
    """The Python entry points: a C++ extension against torch's headers that links to libmadakv.so beside it."""
    header = os.path.join(ROOT, "include", "madakv.h")
    newest = max(os.path.getmtime(NATIVE_SRC), os.path.getmtime(header))
    if force or not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < newest:
        import torch
        from torch.utils import cpp_extension

        inc = cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
        subprocess.check_call(
            ["g++", "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
            + [x for d in inc for x in ("-isystem", d)] + ["-o", NATIVE, NATIVE_SRC, "-L", HERE]
            + [x for d in cpp_extension.library_paths("cuda") for x in ("-L", d)]
            + ["-lmadakv", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"])
    return NATIVE


def build(force=False, verbose=False):
    build_probe(force)
    if not force and not needs_build():
        build_native()
        return LIB
    cmd = [
        "nvcc", "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
        "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(HERE, "csrc"),
        "-o", LIB,
    ] + (["-Xptxas", "-v"] if verbose else []) + sources()
    subprocess.check_call(cmd)
    build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
