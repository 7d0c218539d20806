"""Build libnnv.so in-tree with nvcc for sm_100a (no other architecture, no fallback), and the extension module that
marshals the per-layer calls for Python."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnnv.so")
PYCALL = os.path.join(HERE, "_nnvcall.so")
SOURCES = ["plan.cpp", "scheduler.cpp", "cachefile.cpp", "transform.cu", "exec_kernels.cu", "direct_conv.cu", "wino_small.cu", "wino_layer.cu", "gemm_tc.cu", "exec.cu", "pipeline.cu", "noalloc.cu"]


def sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def needs_build():
    if not os.path.exists(LIB) or not os.path.exists(PYCALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(PYCALL))
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    deps = sources() + [os.path.join(CSRC, "pycall.cpp")] + headers + [os.path.join(ROOT, "include", "nnv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force=False, verbose=False):
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-shared", "-Xcompiler", "-fPIC", "--threads", "0",
           "-gencode", "arch=compute_100a,code=sm_100a",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-shared", "-fPIC", "-Wall",
                           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"),
                           "-o", PYCALL, os.path.join(CSRC, "pycall.cpp"), "-L", HERE, "-l:libnnv.so", "-Wl,-rpath,$ORIGIN"])
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
