"""Builds the CUDA library libofdft_gb300.so in-tree (sm_103a).

The translation units (C-ABI layer, FP32 and FP64 engines, the plane-pass
kernels of each precision, the allocation-free entry point) are compiled in
parallel with nvcc and linked into
paper_2601_23002_gb300/_build/libofdft_gb300.so.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libofdft_gb300.so")
SOURCES = ["api.cu", "engine_f32.cu", "engine_f64.cu", "plane_f32.cu", "plane_f64.cu", "plane2_f32.cu",
           "plane2_f64.cu", "noalloc.cu"]
# sources compiled several times, each part with its own share of the kernels (-DCPASS_PART=i)
PARTED = {"cpass_f32.cu": 6, "cpass_f64.cu": 4}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)
             if f.endswith((".cu", ".cuh", ".h"))]
    files.append(os.path.join(HERE, "..", "include", "ofdft.h"))
    return files


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    os.makedirs(OUT, exist_ok=True)
    nvcc = _nvcc()
    flags = ARCH + ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
                    "-I", os.path.join(HERE, "..", "include")]

    jobs = [(src, part) for src, count in PARTED.items() for part in range(count)]
    jobs += [(src, None) for src in SOURCES]

    def compile_one(job):
        src, part = job
        obj = os.path.join(OUT, src.replace(".cu", ".o" if part is None else f"_{part}.o"))
        define = [] if part is None else [f"-DCPASS_PART={part}"]
        cmd = [nvcc] + flags + define + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stderr[-4000:]}")
        return obj

    with ThreadPoolExecutor(max_workers=len(jobs)) as ex:
        objs = list(ex.map(compile_one, jobs))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs + ["-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr[-4000:]}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
