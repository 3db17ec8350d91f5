"""Builds the CUDA library in-tree with nvcc for sm_100a.

``build()`` compiles every ``csrc/*.cu`` to an object file (in parallel), links
``libdvp_b200.so`` beside this file and compiles ``_host.so``, the Python helper
that lays a call's outputs over one allocation.  Objects are rebuilt only when a
source or header is newer, ``_host.so`` also after a change of interpreter or torch.  Run as ``python -m paper_2512_23087_b200.build``;
``--debug-bounds`` builds the bounds-checking library instead.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libdvp_b200.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _newest_header() -> float:
    hdrs = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    return max(os.path.getmtime(h) for h in hdrs)


HOST = os.path.join(HERE, "_host.so")


def host_target() -> str:
    """What ``_host.so`` has to be built for: it uses torch's C++ classes and this interpreter's, whose layouts differ from
    version to version.  It carries this text, and ``binding.load_library`` refuses one built for something else."""
    import torch
    return f"{sys.implementation.cache_tag} torch {torch.__version__}"


def _host_is_for(target: str) -> bool:
    try:
        with open(HOST, "rb") as f:
            return f"[built for {target}]".encode() in f.read()
    except OSError:
        return False


def build_host(force: bool = False) -> str:
    """The Python helper ``_host`` (g++ against this interpreter's and torch's headers)."""
    src = os.path.join(CSRC, "host_outputs.cpp")
    target = host_target()
    if not force and _host_is_for(target) and os.path.getmtime(HOST) >= max(
            os.path.getmtime(f) for f in (src, os.path.join(ROOT, "include", "dvp.h"))):
        return HOST
    import sysconfig
    import torch
    base = os.path.join(os.path.dirname(torch.__file__))
    nvcc = shutil.which(_nvcc()) or "/usr/local/cuda/bin/nvcc"   # its headers
    tmp = HOST + f".{os.getpid()}.tmp"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", src, "-o", tmp,
           f'-DDVP_HOST_TARGET="{target}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", sysconfig.get_paths()["include"],
           "-isystem", os.path.join(base, "include"),
           "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"),
           "-L", os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed: " + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    os.replace(tmp, HOST)
    return HOST


LIB_BOUNDS = os.path.join(HERE, "libdvp_b200_bounds.so")


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """``debug_bounds``: the second library, compiled with -DDVP_DEBUG_BOUNDS (every index of
    the row kernels' on-chip tables and every global offset checked, reported through
    ``dvp_debug_bounds_status``), as ``libdvp_b200_bounds.so``."""
    obj_dir = OBJ + ("_bounds" if debug_bounds else "")
    lib = LIB_BOUNDS if debug_bounds else LIB
    extra = ["-DDVP_DEBUG_BOUNDS"] if debug_bounds else []
    os.makedirs(obj_dir, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    hdr_time = _newest_header()
    nvcc = _nvcc()
    jobs = []
    objs = []
    for src in srcs:
        obj = os.path.join(obj_dir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        stale = force or not os.path.exists(obj) or \
            os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time)
        if stale:
            cmd = [nvcc, *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        return r.stderr

    if jobs:
        with ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            for log in ex.map(run, jobs):
                if verbose and log:
                    print(log, file=sys.stderr)
    build_host(force and not debug_bounds)
    if jobs or not os.path.exists(lib):
        tmp = lib + f".{os.getpid()}.tmp"
        run([nvcc, "-shared", "-o", tmp, *objs, "-lcudart"])
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug_bounds="--debug-bounds" in sys.argv))
