"""Builds csrc/*.cu into libdp_ghost.so (sm_100a only) and csrc/marshal.cpp into the Python
extension _marshal.so, next to this file.

    python -m paper_2609_40335_b200.build [--force] [--verbose] [--check]

--check also builds libdp_ghost_check.so: the same sources with -DDP_BOUNDS_CHECK (every index a
kernel computes from data is range-checked before the access).  Load it in place of the normal
library by setting DP_GHOST_LIB to its path.

nvcc cross-compiles without a GPU.  The shared library is kept in-tree so that it travels
with the source to the machine that has the GPU.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ_DIR = os.path.join(HERE, "build")
LIB_PATH = os.path.join(HERE, "libdp_ghost.so")
CHECK_LIB_PATH = os.path.join(HERE, "libdp_ghost_check.so")
MARSHAL_PATH = os.path.join(HERE, "_marshal.so")
MARSHAL_STAMP = os.path.join(OBJ_DIR, "marshal.stamp")       # what _marshal.so was compiled with
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC"]


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _headers():
    inc = os.path.join(os.path.dirname(HERE), "include")
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hs += [os.path.join(inc, f) for f in os.listdir(inc)]
    return hs


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    """Compile the library; check=True builds the range-checked variant instead."""
    nvcc = os.environ.get("NVCC", "nvcc")
    obj_dir = os.path.join(OBJ_DIR, "check") if check else OBJ_DIR
    lib_path = CHECK_LIB_PATH if check else LIB_PATH
    extra = ["-DDP_BOUNDS_CHECK"] if check else []
    os.makedirs(obj_dir, exist_ok=True)
    hdrs = _headers()
    jobs = []
    objs = []
    for src in _sources():
        obj = os.path.join(obj_dir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs):
            cmd = [nvcc, *ARCH, *FLAGS, *extra, "-c", src, "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    if not check:
        build_marshal(force)
    with cf.ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode != 0:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {cmd[-3]}")
    if force or jobs or _stale(lib_path, objs):
        cmd = [nvcc, *ARCH, "-shared", "-o", lib_path, *objs]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    return lib_path


def build_marshal(force: bool = False) -> str:
    """Compile the extension that reads the tensors of a call (see csrc/marshal.cpp).  It belongs to the torch and
    the Python it was compiled against: another one of either, or another command, makes it stale as well."""
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    src = os.path.join(CSRC, "marshal.cpp")
    header = os.path.join(os.path.dirname(HERE), "include", "dp_ghost.h")
    lib = os.path.join(root, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DDP_TORCH_VERSION="{torch.__version__}"',
           "-I" + os.path.join(root, "include"), "-I" + sysconfig.get_paths()["include"],
           "-I" + os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"), src, "-o", MARSHAL_PATH,
           "-L" + lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath," + lib]
    made_by = "\n".join([sys.version, torch.__version__, *cmd])
    if not force and not _stale(MARSHAL_PATH, [src, header]) and os.path.exists(MARSHAL_STAMP):
        with open(MARSHAL_STAMP) as f:
            if f.read() == made_by:
                return MARSHAL_PATH
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        raise RuntimeError("compiling marshal.cpp failed")
    os.makedirs(os.path.dirname(MARSHAL_STAMP), exist_ok=True)
    with open(MARSHAL_STAMP, "w") as f:
        f.write(made_by)
    return MARSHAL_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
    if "--check" in sys.argv:
        print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, check=True))
