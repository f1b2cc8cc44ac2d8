"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the
native torch marshalling on top of it.

Every csrc/*.cu is compiled to an object file under _build/ (in parallel, only when stale) and
the objects are linked into libvla.so next to this file; csrc_torch/vla_torch.cpp becomes _vla_torch.so.
"""
from __future__ import annotations

import concurrent.futures
import glob
import importlib.util
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libvla.so")
EXT_SRC = os.path.join(PKG, "csrc_torch", "vla_torch.cpp")
EXT = os.path.join(PKG, "_vla_torch.so")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]


def _obj(src: str) -> str:
    return os.path.join(OBJ, os.path.splitext(os.path.basename(src))[0] + ".o")


def _obj_stale(src: str) -> bool:
    o = _obj(src)
    if not os.path.exists(o):
        return True
    t = os.path.getmtime(o)
    return any(os.path.getmtime(d) > t for d in [src] + _headers())


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in sources() + _headers())


def _build_ext(force: bool) -> None:
    """The marshalling module: links against libvla.so beside it and the torch this interpreter has."""
    deps = [EXT_SRC, os.path.join(ROOT, "include", "vla.h"), os.path.abspath(__file__)]
    if not force and os.path.exists(EXT) and all(os.path.getmtime(d) <= os.path.getmtime(EXT) for d in deps):
        return
    t = os.path.dirname(importlib.util.find_spec("torch").origin)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    tmp = EXT + ".tmp.%d" % os.getpid()
    inc = [os.path.join(ROOT, "include"), t + "/include", t + "/include/torch/csrc/api/include",
           sysconfig.get_paths()["include"], cuda + "/include"]
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-w", "-o", tmp, EXT_SRC] + ["-I" + i for i in inc] +
                          ["-L" + PKG, "-l:libvla.so", "-L" + t + "/lib", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda",
                           "-ltorch", "-ltorch_python", "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, EXT)


def build(force: bool = False, verbose: bool = False, jobs: int = 0) -> str:
    """Compile csrc/*.cu, link libvla.so and _vla_torch.so next to this file; returns the library's path."""
    if not force and not _stale():
        _build_ext(False)
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    todo = [s for s in sources() if force or _obj_stale(s)]

    def compile_one(src: str) -> str:
        tmp = _obj(src) + ".tmp.%d" % os.getpid()
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
            ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", "-o", tmp, src]
        r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed on %s:\n%s" % (src, r.stdout))
        os.replace(tmp, _obj(src))
        return r.stdout

    jobs = jobs or min(len(todo) or 1, os.cpu_count() or 1)
    with concurrent.futures.ThreadPoolExecutor(max_workers=jobs) as pool:
        for out in pool.map(compile_one, todo):
            if verbose and out:
                print(out)
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-Xcompiler", "-fPIC", "-gencode",
                           "arch=compute_100a,code=sm_100a", "-o", tmp] + [_obj(s) for s in sources()])
    os.replace(tmp, LIB)
    _build_ext(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
