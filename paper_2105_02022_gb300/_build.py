"""In-tree build of the native parts: the CUDA library (sm_103a) and the input
generator.  Outputs sit next to their sources and are git-ignored."""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
ROOT = os.path.dirname(PKG)
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build_obj")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
              "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return cand


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(s) > t for s in sources)


def build_graphgen() -> str:
    src = os.path.join(PKG, "graphgen", "graphgen.c")
    out = os.path.join(PKG, "graphgen", "libgraphgen.so")
    if _stale(out, [src]):
        # with OpenMP when the toolchain has it; the output is the same either way
        base = ["gcc", "-O2", "-fPIC", "-shared", "-o", out + ".tmp", src, "-lm"]
        if subprocess.run(base[:1] + ["-fopenmp"] + base[1:], capture_output=True).returncode != 0:
            subprocess.check_call(base)
        os.replace(out + ".tmp", out)
    return out


def lib_path() -> str:
    return os.path.join(PKG, "libkmp.so")


def build_kmp(verbose: bool = False, extra=()) -> str:
    """Compile every csrc/*.cu for sm_103a (in parallel) and link libkmp.so."""
    os.makedirs(BUILD, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    hdrs = sorted(h for pat in (os.path.join(CSRC, "*.cuh"), os.path.join(CSRC, "*.h"), os.path.join(INCLUDE, "*.h"))
                  for h in glob.glob(pat))
    out = lib_path()
    nvcc = _nvcc()
    objs = []

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        with open(src) as f:  # a second build of another source includes it
            text = f.read()
        included = [x for x in srcs if f'#include "{os.path.basename(x)}"' in text]
        if _stale(obj, [src] + included + hdrs):
            cmd = [nvcc, *ARCH, *NVCC_FLAGS, *extra, "-c", src, "-o", obj + ".tmp"]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            r = subprocess.run(cmd, capture_output=True, text=True)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr}")
            if verbose and r.stderr:
                print(r.stderr)
            os.replace(obj + ".tmp", obj)
        return obj

    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(srcs), os.cpu_count() or 4))) as ex:
        objs = list(ex.map(compile_one, srcs))
    if _stale(out, objs):
        cmd = [nvcc, *ARCH, "-shared", "-o", out + ".tmp", *objs, "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stderr}")
        os.replace(out + ".tmp", out)
    return out


def build_all(verbose: bool = False) -> None:
    build_graphgen()
    build_kmp(verbose=verbose)
