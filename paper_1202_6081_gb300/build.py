"""Build liblbm.so, the C-ABI CUDA library, in-tree for sm_103a.

The translation units (csrc/kernels.cu once per lattice, storage type and
group of kernels) are compiled by nvcc in parallel, then linked into
paper_1202_6081_gb300/liblbm.so (CUDA runtime linked statically).  Run ``python -m paper_1202_6081_gb300.build`` or call
``build()``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "liblbm.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# translation units: (object name, source, macro definitions); the slowest first
UNITS = [("kernels_%s_q%d_%s" % (group.lower(), Q, name), "kernels.cu",
          ["-DLBM_GROUP=" + group, "-DLBM_Q=%d" % Q, "-DLBM_T=" + T])
         for group in ("STEP", "ADJOINT", "INPLACE", "STATE") for Q in (27, 15)
         for name, T in (("f32", "float"), ("f16", "__half"), ("bf16", "__nv_bfloat16"))]
UNITS += [("reduce", "reduce.cu", []), ("api", "api.cu", [])]


def nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build liblbm.so")
    return path


def _flags(verbose_ptxas: bool):
    f = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
    f += ARCH
    if verbose_ptxas:
        f += ["-Xptxas", "-v"]
    return f


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, n) for n in os.listdir(CSRC)]
    deps.append(os.path.join(INCLUDE, "lbm.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose_ptxas: bool = False, quiet: bool = True) -> str:
    """Compile (if stale) and return the path of liblbm.so."""
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    flags = _flags(verbose_ptxas)

    def compile_one(unit):
        name, src, defines = unit
        obj = os.path.join(BUILD, name + ".o")
        cmd = [cc, "-c", os.path.join(CSRC, src), "-o", obj] + defines + flags
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (name, r.stdout, r.stderr))
        return obj, r.stderr

    with ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
        results = list(ex.map(compile_one, UNITS))
    objs = [o for o, _ in results]
    if verbose_ptxas or not quiet:
        for _, log in results:
            sys.stderr.write(log)
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [cc, "-shared", "-o", tmp] + objs + ARCH + ["-Xcompiler", "-fPIC"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv, quiet=False))
