"""Builds the C-ABI CUDA library (sm_100a only) next to this file.

    python -m paper_2603_20586_b200.build [--force]

nvcc cross-compiles without a GPU.  The runtime is linked statically, so the library loads on a
machine without a CUDA driver (every compute entry point then returns MKA_ERR_CUDA).
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmka_b200.so")
HOST_SRC = os.path.join(CSRC, "host_args.cpp")
OBJ_DIR = os.path.join(HERE, "_build")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-DMKA_NO_FAST_MATH",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def host_module() -> str:
    """Path of the binding's argument marshalling (host only).  It is compiled against torch's and Python's headers, so each of their
    versions has a file of its own: one that was built for others is neither loaded nor taken for up to date."""
    import torch
    return os.path.join(HERE, f"_host_args.{sys.implementation.cache_tag}.torch-{torch.__version__}-{str(torch.version.git_version)[:8]}.so")


def _host_module_cmd(out):
    import sysconfig

    import torch
    from torch.utils.cpp_extension import include_paths, library_paths
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include")]
    for path in include_paths():
        cmd += ["-isystem", path]
    for path in library_paths():
        cmd += ["-L", path]
    return cmd + [HOST_SRC, "-o", out, "-lc10", "-ltorch_cpu", "-ltorch_python"]


def build(force: bool = False, verbose: bool = False) -> str:
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    os.makedirs(OBJ_DIR, exist_ok=True)
    objs, jobs = [], []
    for src in _sources():
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("build failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + f".{os.getpid()}.tmp"
        run([NVCC, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp] + objs + ["-cudart", "static"])
        os.replace(tmp, LIB)
    host = host_module()
    if force or _stale(host, [HOST_SRC] + glob.glob(os.path.join(ROOT, "include", "*.h"))):
        tmp = host + f".{os.getpid()}.tmp"
        run(_host_module_cmd(tmp))
        os.replace(tmp, host)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
