"""Compile the CUDA sources into the in-tree shared library libgbgemm.so.

Every translation unit is compiled for sm_103a only (one -gencode), in
parallel, then linked with ``nvcc -shared``.  The result lands in
``paper_1608_05265_gb300/_build/libgbgemm.so`` (git-ignored).  A rebuild is
skipped when the library is newer than every source and header.
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
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libgbgemm.so")
SOURCES = ["api.cu", "simt.cu", "split.cu", "noalloc.cu", "grouped.cu", "tuner.cu", "mlp.cu", "check.cu",
           "gemv.cu", "lu.cu", "direct.cu"]
# Sources compiled once per set of macros (object name, source, macros).
VARIANTS = [(f"direct_inst_p{p}_m{m}", "direct_inst.cu", [f"-DGBG_PARTS={p}", f"-DGBG_MODE_A={m}"])
            for p in (2, 3) for m in (0, 1, 2)]
HEADERS = [os.path.join(CSRC, h) for h in ("internal.h", "split_device.cuh", "simt_device.cuh", "gemm_kernel.cuh",
                                            "grouped.h", "tuner.h", "mlp.h", "direct.h", "direct_kernel.cuh")] + \
    [os.path.join(ROOT, "include", "gbgemm.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "-Xptxas", "-v",
         "-I" + os.path.join(ROOT, "include")]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build libgbgemm.so")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES + [v[1] for v in VARIANTS]] + \
        [h for h in HEADERS if os.path.exists(h)] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(OUT, exist_ok=True)
    cc = nvcc()

    def compile_one(job) -> str:
        name, src, macros = job
        obj = os.path.join(OUT, name + ".o")
        cmd = [cc] + ARCH + FLAGS + macros + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        with open(os.path.join(OUT, name + ".ptxas"), "w") as f:  # registers, spills and shared memory of every kernel
            f.write(r.stderr)
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    jobs = VARIANTS + [(src[:-3], src, []) for src in SOURCES]  # the longest first
    with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
        objs = list(ex.map(compile_one, jobs))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [cc] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
