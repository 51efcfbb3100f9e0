"""Build liblgf.so (the C-ABI library) in-tree with nvcc for sm_103a.

Each translation unit under ``csrc/`` is compiled in parallel to an object
file in ``_build/`` and the objects are linked into ``liblgf.so`` next to
this file.  Only nvcc and the CUDA runtime are needed (no torch, no cmake),
so the same build runs on the x86 build host and on the aarch64 GPU host.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "liblgf.so")
SOURCES = ["k_links.cu", "k_links_fx.cu", "k_gauge_rep.cu", "k_fft.cu", "k_fft_any.cu", "k_fft_fx.cu", "k_fft_long.cu", "k_zt_pairs.cu", "k_fft_axis.cu", "k_fft_plane.cu", "k_fft_zt.cu", "k_warm.cu", "k_tail.cu", "lgf_api.cu", "lgf_noalloc.cu"]
# sources compiled once per part, with -D<macro>=<part>
PARTS = {"k_fft_any.cu": ("LGF_ANY_PART", range(2)),
         "k_fft_fx.cu": ("LGF_FX_PART", range(5)),
         "k_fft_long.cu": ("LGF_LONG_T", ("double", "float")),
         "k_zt_pairs.cu": ("LGF_PAIR_Z", (4, 6, 8, 10, 12, 16, 18, 20, 24, 30, 32, 36, 40, 48, 64))}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: set NVCC or put the CUDA toolkit on PATH")


def _newer(target: str, deps) -> bool:
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(d) <= t for d in deps)


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return hs + [os.path.join(ROOT, "include", "lgf.h")]


def build(verbose: bool = False, extra_flags=()) -> str:
    """Compile (if stale) and return the path of liblgf.so."""
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    hdrs = _headers()
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        macro, parts = PARTS.get(src, (None, (0,)))
        for part in parts:
            o = os.path.join(BUILD, src.replace(".cu", f"_{part}.o" if macro else ".o"))
            objs.append(o)
            if not _newer(o, [s] + hdrs):
                jobs.append([cc, *ARCH, *FLAGS, *extra_flags, *([f"-D{macro}={part}"] if macro else []), "-c", s, "-o", o])

    def run(cmd):
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed ({' '.join(cmd)}):\n{r.stdout}\n{r.stderr}")
        if verbose and (r.stdout or r.stderr):
            print(r.stdout + r.stderr, flush=True)

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(len(jobs), 2 * (os.cpu_count() or 8))) as ex:
            list(ex.map(run, jobs))
    if jobs or not _newer(LIB, objs):
        tmp = LIB + ".tmp"
        run([cc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv))
