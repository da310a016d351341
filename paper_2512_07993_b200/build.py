"""Builds ``libskipkv.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_native.so`` (the Python entry
points over it) with the host compiler."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libskipkv.so")
EXT = os.path.join(HERE, "_native.so")
EXT_SRC = os.path.join(CSRC, "pyext.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17", "--use_fast_math",
         "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def built_for() -> str:
    """The Python and torch that ``_native.so`` is built for: it unpacks their objects, whose layout belongs to one version each."""
    import torch
    return f"python {sys.version_info[0]}.{sys.version_info[1]}, torch {torch.__version__}"


def source_hash() -> str:
    """Content hash of everything the two files are built from (mtimes do not survive a copy)."""
    import hashlib
    h = hashlib.sha256((" ".join(FLAGS[:8]) + built_for()).encode())
    deps = sources() + [EXT_SRC] + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + sorted(glob.glob(os.path.join(ROOT, "include", "*.h")))
    for p in deps:
        h.update(os.path.basename(p).encode())
        h.update(open(p, "rb").read())
    return h.hexdigest()


def stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(EXT) or not os.path.exists(LIB + ".hash"):
        return True
    return open(LIB + ".hash").read().strip() != source_hash()


def _ext_command(out: str):
    """Host compiler command of the extension: it unpacks torch tensors, so it is built against this torch."""
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    inc = [sysconfig.get_paths()["include"], os.path.join(ROOT, "include"), os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"),
           *cpp_extension.include_paths()]
    torch_lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DSKIPKV_BUILT_FOR="{built_for()}"', *(f"-I{d}" for d in inc), EXT_SRC, "-o", out,
            f"-L{HERE}", "-l:libskipkv.so", "-Wl,-rpath,$ORIGIN", f"-L{torch_lib}", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not stale():
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(f"== {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([NVCC, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"], check=True)
    os.replace(tmp, LIB)
    tmp = EXT + f".tmp{os.getpid()}"
    subprocess.run(_ext_command(tmp), check=True)
    os.replace(tmp, EXT)
    with open(LIB + ".hash", "w") as f:
        f.write(source_hash())
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
