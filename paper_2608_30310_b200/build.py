"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgdn_tail_replay.so")
SOURCES = ["api.cu", "sched.cu", "gdn_simt.cu", "gdn_tc.cu", "gdn_decode.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
]


NATIVE = os.path.join(PKG, "_native.so")
NATIVE_SRC = os.path.join(CSRC, "native.cpp")


def build_native(force: bool = False) -> str:
    """Compile the binding's argument path (a CPython extension on torch's C++ tensors; host code only), for the torch and Python at hand."""
    import sysconfig
    import torch
    deps = [NATIVE_SRC, os.path.join(ROOT, "include", "gdn_tail_replay.h")]
    stamp, built_for = os.path.join(ROOT, "build", "native.txt"), "%s %s" % (torch.__version__, sys.version)
    if not force and os.path.exists(NATIVE) and all(os.path.getmtime(d) <= os.path.getmtime(NATIVE) for d in deps) and \
            os.path.exists(stamp) and open(stamp).read() == built_for:
        return NATIVE
    from torch.utils.cpp_extension import include_paths
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    inc = [x for d in include_paths("cuda") + [sysconfig.get_paths()["include"]] for x in ("-isystem", d)]
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
                           '-DBUILT_FOR_TORCH="%s"' % torch.__version__, "-I", os.path.join(ROOT, "include"),
                           *inc, NATIVE_SRC, "-o", tmp, "-L" + lib, "-Wl,-rpath," + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, NATIVE)
    os.makedirs(os.path.dirname(stamp), exist_ok=True)
    with open(stamp, "w") as f:
        f.write(built_for)
    return NATIVE


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "native.cpp"] + [os.path.join(ROOT, "include", "gdn_tail_replay.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libgdn_tail_replay.so (objects under build/), and the binding's extension."""
    build_native(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    bdir = os.path.join(ROOT, "build")
    os.makedirs(bdir, exist_ok=True)
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c",
               os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if out.strip() and (verbose or pr.returncode != 0):
            sys.stderr.write("[%s]\n%s\n" % (src, out))
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs,
                           "-Xcompiler", "-fvisibility=hidden", "-cudart", "static"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
