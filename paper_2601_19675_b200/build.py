"""Builds liblopro.so (the C-ABI CUDA library) for sm_100a with nvcc, and _binding.so (the CPython extension that
marshals arguments for it) with the host compiler, in-tree.

Usage:  python -m paper_2601_19675_b200.build [--force]
Both are written next to this file; the library links the CUDA runtime statically and does not
depend on the driver library at load time, so it can be loaded (not run) on a machine without
a GPU.  The library needs no torch; without one it is built alone.
"""
from __future__ import annotations

import importlib.metadata
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblopro.so")
BINDING = os.path.join(HERE, "_binding.so")
STAMP = os.path.join(HERE, "_build", "binding.txt")
SOURCES = ["api.cu", "pack.cu", "rotate.cu", "decode.cu", "stream.cu", "tall.cu", "warps.cu", "noalloc.cu", "prefill.cu", "lowrank.cu", "rowblock.cu", "quantize.cu", "sketch.cu", "block.cu", "vq.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc():
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _torch_version():
    try:
        return importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None


def _binding_for():
    """What the extension is compiled against: it is good for this Python and this torch only."""
    return f"{sys.implementation.cache_tag} torch {_torch_version()}"


def _stale():
    if not os.path.exists(LIB) or not os.path.exists(BINDING):
        return True
    if os.path.exists(STAMP):
        with open(STAMP) as f:
            if f.read() != _binding_for():
                return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    inc = os.path.join(ROOT, "include")
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(inc, f) for f in os.listdir(inc)] + [__file__]
    return any(os.path.getmtime(d) > t for d in deps)


def _binding_command():
    import sysconfig

    import torch
    th = os.path.dirname(torch.__file__)
    cuda_home = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    inc = [os.path.join(th, "include"), os.path.join(th, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda_home, "include")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-I", os.path.join(ROOT, "include"),
            "-I", sysconfig.get_paths()["include"], *[a for d in inc for a in ("-isystem", d)],
            os.path.join(CSRC, "binding.cpp"), "-o", BINDING, "-L", os.path.join(th, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force=False, verbose=False):
    """Compile every .cu of the library for sm_100a and link liblopro.so; compile the binding."""
    if not force and not _stale():
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    objs = []
    procs = []
    if _torch_version() is None:
        sys.stderr.write("torch is not installed: liblopro.so is built without the Python extension\n")
    else:
        procs.append(("binding.cpp", subprocess.Popen(_binding_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for src in SOURCES:
        obj = os.path.join(objdir, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError(f"the compiler failed on {src}")
    cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs]
    subprocess.run(cmd, check=True)
    if _torch_version() is not None:
        with open(STAMP, "w") as f:
            f.write(_binding_for())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
