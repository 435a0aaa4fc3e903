"""Builds in-tree: the CUDA library paper_2504_00492_b200/libpf.so (sm_100a only) and the extension _pf_ext.so through which
the Python entry points call it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libpf.so")
EXT_SRC = os.path.join(CSRC, "pf_ext.cpp")
EXT = os.path.join(PKG, "_pf_ext.so")
EXT_TAG = os.path.join(PKG, "_build", "_pf_ext.tag")      # what EXT was built against

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "--extended-lambda",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _ext_stale(tag: str) -> bool:
    deps = [EXT_SRC, os.path.join(ROOT, "include", "pf.h")]
    if not os.path.exists(EXT) or any(os.path.getmtime(d) > os.path.getmtime(EXT) for d in deps):
        return True
    try:
        with open(EXT_TAG) as f:
            return f.read() != tag
    except OSError:
        return True


def build_ext(force: bool = False) -> str:
    """Compile the call path of the Python entry points against the installed torch's headers (and again when another torch or
    Python is installed: the extension is tied to their ABI)."""
    import sysconfig

    import torch
    tag = f"torch {torch.__version__} abi {int(torch._C._GLIBCXX_USE_CXX11_ABI)} python {sysconfig.get_config_var('SOABI')}"
    if not force and not _ext_stale(tag):
        return EXT
    t = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = EXT + ".tmp%d" % os.getpid()
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
                    f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(t, "include"),
                    "-isystem", os.path.join(t, "include", "torch", "csrc", "api", "include"),
                    "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"),
                    EXT_SRC, "-o", tmp, "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu",
                    "-lc10_cuda", "-lc10"], check=True)
    os.replace(tmp, EXT)
    os.makedirs(os.path.dirname(EXT_TAG), exist_ok=True)
    with open(EXT_TAG, "w") as f:
        f.write(tag)
    return EXT


def build(force: bool = False, verbose: bool = False, extra_flags=(), out: str = None) -> str:
    """Compile every .cu under csrc/ and link libpf.so.  Returns the library path.
    extra_flags / out: a diagnostic build (e.g. ("-DPF_ENDS",)) into another file, objects kept apart."""
    if out is None:
        build_ext(force)
        if not force and not _stale():
            return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    objs = []
    bdir = os.path.join(PKG, "_build" if out is None else "_build_diag")
    os.makedirs(bdir, exist_ok=True)
    procs = []
    for src in sources():
        obj = os.path.join(bdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, *extra_flags, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd)))
    for src, pr in procs:
        if pr.wait() != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    target = LIB if out is None else out
    tmp = target + ".tmp%d" % os.getpid()
    subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs], check=True)
    os.replace(tmp, target)
    return target


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
