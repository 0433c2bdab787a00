"""In-tree build of libpp.so (CUDA C++ for sm_103a) with nvcc only."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libpp.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpp")


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def units():
    """(source, defines, object) of every translation unit: one for each csrc/*.cu, and
    one for each length of the two that are compiled length by length."""
    lengths = {}
    with open(os.path.join(CSRC, "pp_lines_lengths.h")) as f:
        for block in f.read().split("#define ")[1:]:
            lengths[block.split("(")[0]] = re.findall(r"X\((\d+), (\d+), (\d+)\)", block)
    each = {"pp_lines_unit.cu": "PP_LINE_LENGTHS", "pp_cart_unit.cu": "PP_CART_LENGTHS"}
    out = []
    # the longest lengths first: their kernels take the longest to compile
    for name, group in each.items():
        for n, n1, n2 in sorted(lengths[group], key=lambda t: -int(t[0])):
            out.append((os.path.join(CSRC, name), ["-DPP_N1=" + n1, "-DPP_N2=" + n2],
                        os.path.join(BUILD, "%s_%s.o" % (name[:-3], n))))
    whole = [s for s in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if os.path.basename(s) not in each]
    return [(s, [], os.path.join(BUILD, os.path.basename(s)[:-3] + ".o")) for s in whole] + out


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every csrc/*.cu in parallel and link libpp.so; returns its path."""
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    deps = srcs + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest(deps):
        return LIB
    jobs = units()
    objs = [obj for _, _, obj in jobs]

    def compile_one(job):
        src, defines, obj = job
        cmd = [nvcc, *ARCH, *FLAGS, *defines, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s%s" % (src, r.stdout, r.stderr))
        if verbose:
            print(" ".join(cmd))
        return obj

    with ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 1))) as ex:
        list(ex.map(compile_one, jobs))
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "static"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
