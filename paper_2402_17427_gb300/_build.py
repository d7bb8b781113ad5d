"""Builds the CUDA library libvgrast.so in-tree (nvcc, sm_103a only).

Each .cu file is compiled in parallel with ``-gencode arch=compute_103a,code=sm_103a`` and the
objects are linked into ``paper_2402_17427_gb300/libvgrast.so`` (CUDA runtime linked
statically, so the library needs only the driver at run time).  Where torch and its headers are
installed, the autograd nodes of the torch front end (``csrc/front.cpp``, host code) become ``_vgfront.so``;
they are made again when the installed torch or Python is another than they were compiled against.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libvgrast.so")
FRONT_SRC = os.path.join(CSRC, "front.cpp")
FRONT = os.path.join(PKG, "_vgfront.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "-I" + INCLUDE, "-I" + CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libvgrast.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _stale_lib() -> bool:
    return _older(LIB, sources() + [h for d, e in ((CSRC, "h"), (CSRC, "cuh"), (INCLUDE, "h"))
                                    for h in glob.glob(os.path.join(d, "*." + e))])


def front_torch():
    """The installed torch if the front end's nodes can be compiled against it, else None."""
    try:
        import torch
    except ImportError:
        return None
    header = os.path.join(os.path.dirname(torch.__file__), "include", "torch", "csrc", "autograd", "custom_function.h")
    return torch if os.path.exists(header) else None


def front_key(torch) -> str:
    """What _vgfront.so depends on besides its sources: a C++ ABI that the versions of torch and Python decide.
    The library carries it as a string."""
    return (f"vgfront for torch {torch.__version__}, cxx11 {int(torch._C._GLIBCXX_USE_CXX11_ABI)}, "
            f"{sysconfig.get_config_var('SOABI')};")


def front_matches(torch) -> bool:
    """Whether the _vgfront.so that is there was compiled against this torch."""
    with open(FRONT, "rb") as f:
        return front_key(torch).encode() in f.read()


def _stale_front(torch) -> bool:
    return _older(FRONT, [FRONT_SRC, *glob.glob(os.path.join(INCLUDE, "*.h"))]) or not front_matches(torch)


def build_front(torch) -> None:
    """Compiles the autograd nodes with the host compiler against the installed torch."""
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc())))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"], INCLUDE]
    tmp = FRONT + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DVG_FRONT_KEY="{front_key(torch)}"', *[f"-I{d}" for d in inc], FRONT_SRC,
           "-o", tmp, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed on {FRONT_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, FRONT)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OUT_DIR, exist_ok=True)
    torch = front_torch()
    with cf.ThreadPoolExecutor(max_workers=min(9, os.cpu_count() or 4)) as ex:
        front = ex.submit(build_front, torch) if torch and (force or _stale_front(torch)) else None
        if force or _stale_lib():
            _build_lib(ex, verbose)
        if front:
            front.result()      # the library stands whatever becomes of the nodes
    return LIB


def _build_lib(ex, verbose: bool) -> None:
    cc = nvcc()

    def compile_one(src):
        obj = os.path.join(OUT_DIR, os.path.basename(src).replace(".cu", ".o"))
        cmd = [cc, *ARCH, *FLAGS, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr)
        return obj

    objs = list(ex.map(compile_one, sources()))
    tmp = LIB + f".tmp{os.getpid()}"
    r = subprocess.run([cc, *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)


if __name__ == "__main__":
    print(build(force=True, verbose=True))
