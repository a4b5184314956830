"""Build libmcg.so (the C-ABI CUDA library) in-tree for sm_103a.

Each .cu file is compiled to an object in parallel, then linked into
`paper_0807_0264_gb300/_lib/libmcg.so` with the CUDA runtime linked
statically.  Run `python -m paper_0807_0264_gb300.build` or call build().
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_lib")
LIB = os.path.join(OUT_DIR, "libmcg.so")
SOURCES = ["mcg_capi.cu", "mcg_field.cu", "mcg_field_fx.cu", "mcg_observables.cu", "mcg_smear.cu", "mcg_smear_fx.cu",
           "mcg_smear_bwd_fx.cu", "mcg_sweep.cu", "mcg_sweep_f32.cu", "mcg_sweep_fx.cu", "mcg_sweep_df.cu",
           "mcg_wilson_fx.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _flags(extra=()):
    return ["-std=c++17", "-O3", "-lineinfo", *ARCH, "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
            "-I", os.path.join(HERE, "..", "include"), *extra]


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False, check: bool = False) -> str:
    """Build libmcg.so, or with check=True the index-checking variant
    libmcg_check.so (every kernel compiled with -DMCG_CHECK; objects in
    _lib/check) that mcg.py loads when MCG_LIBRARY names it."""
    if check:
        return _build(os.path.join(OUT_DIR, "check"), LIB_CHECK, ["-DMCG_CHECK"], force, verbose, ptxas_info)
    return _build(OUT_DIR, LIB, [], force, verbose, ptxas_info)


LIB_CHECK = os.path.join(OUT_DIR, "libmcg_check.so")


def _build(out_dir, lib, defines, force, verbose, ptxas_info) -> str:
    os.makedirs(out_dir, exist_ok=True)
    headers = [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith((".cuh", ".h"))]
    headers.append(os.path.join(HERE, "..", "include", "mcg.h"))
    objs = []
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(out_dir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s, *headers]):
            extra = ["-Xptxas", "-v"] if ptxas_info else []
            jobs.append([nvcc(), *_flags([*defines, *extra]), "-c", s, "-o", o])
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
            results = list(ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs))
        for cmd, r in zip(jobs, results):
            if verbose or ptxas_info or r.returncode:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode:
                raise RuntimeError(f"nvcc failed: {' '.join(cmd)}")
    if force or jobs or _stale(lib, objs):
        tmp = lib + f".tmp{os.getpid()}"
        r = subprocess.run([nvcc(), *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
        if r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError(f"link of {os.path.basename(lib)} failed")
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv,
                check="--check" in sys.argv))
