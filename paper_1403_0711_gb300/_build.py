"""In-tree build of libcoulps.so for sm_103a (nvcc, no cmake).

Each .cu file is compiled to an object in parallel, then linked into
``paper_1403_0711_gb300/libcoulps.so`` (CUDA runtime linked statically, so the
library does not depend on the runtime that the Python framework ships).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
LIB = PKG / "libcoulps.so"
BUILD = PKG.parent / "_build"

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVFLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-O2", "--expt-relaxed-constexpr",
           "-I", str(CSRC), "-I", str(INCLUDE), "-I", str(BUILD)]
SOURCES = ["sweep.cu", "pass_fused.cu", "pass_pair.cu", "resident.cu", "measure.cu", "api.cu", "measure_static.cu", "batch.cu",
           "cv_conv.cu", "cv_ops.cu", "cv_train.cu", "gcv.cu", "batch_gcv.cu", "sor.cu"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and Path(cand).exists():
            return cand
    raise RuntimeError("nvcc not found")


def _stale() -> bool:
    if not LIB.exists():
        return True
    t = LIB.stat().st_mtime
    deps = list(CSRC.glob("*")) + list(INCLUDE.glob("*.h")) + [Path(__file__)]
    return any(p.stat().st_mtime > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> Path:
    if not force and not _stale():
        return LIB
    BUILD.mkdir(exist_ok=True)
    nv = nvcc()
    # the FP64 deviate's table, included by device_common.cuh (about a second)
    subprocess.run([sys.executable, str(CSRC / "gen_erfcinv_f64.py"),
                    str(BUILD / "erfcinv_f64_table.inc")], check=True)

    def compile_one(src):
        obj = BUILD / (Path(src).stem + ".o")
        cmd = [nv, *ARCH, *NVFLAGS, "-c", str(CSRC / src), "-o", str(obj)]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    if verbose:
        for _, log in results:
            print(log)
    tmp = LIB.with_suffix(f".{os.getpid()}.tmp")
    cmd = [nv, *ARCH, "-shared", "-o", str(tmp), *[str(o) for o, _ in results],
           "-cudart=static"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
