"""Build libmxq.so (hand-written CUDA for sm_100a) in-tree with nvcc, and the extension module _native with g++.

``python -m paper_2605_08565_b200.build [--force] [--verbose]``

Every ``csrc/*.cu`` is compiled to an object file in ``_build/`` (in parallel) and linked into
``paper_2605_08565_b200/libmxq.so``.  No fast-math, no flush-to-zero, no FMA contraction: the
kernels must reproduce IEEE binary32 results bit for bit.  ``csrc/mxq_python.cpp``, which unpacks the arguments of the
binding's inner-loop calls, is compiled against the installed torch to ``paper_2605_08565_b200/_native.<versions>.so``; where that fails (no g++, no
headers of Python or torch) the library is complete without it and the binding uses ctypes.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libmxq.so")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-fmad=false", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: libmxq cannot be built")
    return exe


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def native_path() -> str:
    """The extension module's file.  It holds the layouts of torch's tensors and of Python's objects, so its name carries both versions:
    another torch or Python finds no module, not this one."""
    import torch
    return os.path.join(HERE, f"_native.torch{torch.__version__}{sysconfig.get_config_var('EXT_SUFFIX')}")


def build_native(force: bool = False, verbose: bool = False) -> str:
    src = os.path.join(CSRC, "mxq_python.cpp")
    target = native_path()
    if not force and not _stale(target, [src, os.path.join(os.path.dirname(HERE), "include", "mxq.h"), os.path.abspath(__file__)]):
        return target
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    tmp = target + f".{os.getpid()}.tmp"
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(f"-I{d}" for d in include), src, "-o", tmp,
           "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("build of the extension module _native failed")
    os.replace(tmp, target)
    return target


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        [os.path.join(os.path.dirname(HERE), "include", "mxq.h"), os.path.abspath(__file__)]
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    nvcc = _nvcc()
    jobs = []
    objs = []
    for src in sources:
        obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            cmd = [nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), "-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
            for cmd, r in ex.map(run, jobs):
                if verbose or r.returncode != 0:
                    sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
                if r.returncode != 0:
                    raise RuntimeError(f"nvcc failed for {cmd[-3]}")
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + f".{os.getpid()}.tmp"
        r = subprocess.run([nvcc, "-shared", "-o", tmp, *objs, "-Xcompiler", "-fPIC"], capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link of libmxq.so failed")
        os.replace(tmp, LIB)
    try:
        build_native(force, verbose)
    except (RuntimeError, OSError) as e:
        warnings.warn(f"{e}: the binding goes through ctypes", RuntimeWarning, stacklevel=2)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
