"""Builds the C-ABI CUDA library in-tree, paper_2609_09721_b200/libefq_b200.so (sm_100a only), and the CPython extension
beside it that calls it, efq_fastcall.so."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libefq_b200.so")
FASTCALL_SRC = os.path.join(CSRC, "fastcall.c")
FASTCALL = os.path.join(_HERE, "efq_fastcall.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
         "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(FASTCALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(FASTCALL))
    deps = sources() + [FASTCALL_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    objs = []
    os.makedirs(os.path.join(_HERE, "build"), exist_ok=True)
    procs = []
    for src in sources():
        obj = os.path.join(_HERE, "build", os.path.basename(src)[:-3] + ".o")
        cmd = [NVCC, *FLAGS, "-c", src, "-o", obj] + (["-Xptxas", "-v"] if verbose else [])
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([NVCC, "-shared", "-o", tmp, *objs, "-lcuda", "-cudart", "static"], check=True)
    os.replace(tmp, LIB)
    tmp = FASTCALL + f".tmp{os.getpid()}"
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(ROOT, "include"), FASTCALL_SRC, "-o", tmp], check=True)
    os.replace(tmp, FASTCALL)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
