"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a.

    python -m paper_2412_18106_b200.build [--force]

The shared object lands beside this file (libxy_attn.so); nvcc cross-compiles
without a GPU and without torch.  The binding's native calls (_fastcall.so, a CPython
extension against torch's headers) are compiled beside it with the host compiler, where
torch is installed, and again when its version changes.
"""
from __future__ import annotations

import glob
import importlib.metadata
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libxy_attn.so")
FASTCALL = os.path.join(HERE, "_fastcall.so")
FASTCALL_STAMP = os.path.join(HERE, "build", "fastcall.torch")  # the torch version it was compiled against

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cc")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(ROOT, "include", "*.h"))
    for pat in ("*.h", "*.cuh", "*.inc"):
        deps += glob.glob(os.path.join(CSRC, pat))
    return any(os.path.getmtime(d) > t for d in deps)


def torch_version():
    """The installed torch's version (torch is not imported), or None."""
    try:
        return importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None


def _fastcall_stale() -> bool:
    if not os.path.exists(FASTCALL) or not os.path.exists(FASTCALL_STAMP):
        return True
    with open(FASTCALL_STAMP) as f:
        if f.read() != torch_version():
            return True
    deps = [os.path.join(CSRC, "fastcall.cpp")] + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > os.path.getmtime(FASTCALL) for d in deps)


def start_fastcall():
    """Starts the compiler on the CPython extension; returns (process, temporary output)."""
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = FASTCALL + ".tmp.%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-w",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-I", os.path.join(ROOT, "include"), "-I", inc, "-I", os.path.join(inc, "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", "/usr/local/cuda/include",
           os.path.join(CSRC, "fastcall.cpp"), "-o", tmp, "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT), tmp


def build(force: bool = False, verbose: bool = False) -> str:
    fast = None
    if torch_version() is None:
        sys.stderr.write("torch is not installed: building the C library only\n")
    elif force or _fastcall_stale():
        try:
            fast = start_fastcall()
        except Exception as e:  # the library is built all the same
            fast = e
    try:
        return _build_lib(force, verbose)
    finally:
        if isinstance(fast, Exception):
            raise RuntimeError("compiling fastcall.cpp failed") from fast
        if fast is not None:
            out = fast[0].communicate()[0].decode()
            if fast[0].returncode != 0:
                raise RuntimeError("compiling fastcall.cpp failed:\n" + out[-3000:])
            os.replace(fast[1], FASTCALL)
            os.makedirs(os.path.dirname(FASTCALL_STAMP), exist_ok=True)
            with open(FASTCALL_STAMP, "w") as f:
                f.write(torch_version())


def _build_lib(force: bool, verbose: bool) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    procs, objs = [], []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src) + ".o")
        objs.append(obj)
        extra = ["-DXY_ENABLE_TRACE"] if os.environ.get("XY_BUILD_TRACE") == "1" else []
        extra += os.environ.get("XY_NVCC_EXTRA", "").split()
        cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-x", "cu", "-c", src, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = False
    for src, p in procs:
        out = p.communicate()[0].decode()
        if p.returncode != 0 or verbose:
            sys.stderr.write("== %s\n%s\n" % (os.path.basename(src), out))
        failed = failed or p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp]
                          + objs + ["-cudart", "static"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
