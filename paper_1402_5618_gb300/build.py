"""Build the CUDA library ``libppcweno.so`` for sm_103a with nvcc.

Every translation unit under ``csrc/`` is compiled in parallel into
``_build/`` and linked into one shared library exposing the C ABI of
``include/pp_cweno.h``.  Nothing is installed outside the package folder.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libppcweno.so")
SOURCES = ["pp_cweno.cu", "sweep_f64_m8.cu", "sweep_f64_m16.cu", "sweep_f32_m8.cu",
           "sweep_f32_m16.cu", "sweep_f64_short.cu", "sweep_f32_short.cu", "char_recon_f64.cu",
           "char_recon_f32.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "-I" + os.path.join(ROOT, "include")]


# the FP32 form uses approximate division / square root and flushes
# denormals; the error-free transformations of the compensated sums use
# explicitly rounded intrinsics, so they are unaffected
FILE_FLAGS = {"sweep_f32_m8.cu": ["--use_fast_math"], "sweep_f32_m16.cu": ["--use_fast_math"],
              "sweep_f32_short.cu": ["--use_fast_math"], "char_recon_f32.cu": ["--use_fast_math"]}


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps() -> list[str]:
    out = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    out.append(os.path.join(ROOT, "include", "pp_cweno.h"))
    return out


def build(force: bool = False, verbose: bool = False, extra: list[str] | None = None) -> str:
    os.makedirs(BUILD, exist_ok=True)
    newest = max(os.path.getmtime(p) for p in _deps())
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= newest:
        return LIB
    nvcc = _nvcc()
    extra = list(extra or [])

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        per_file = FILE_FLAGS.get(src, [])
        cmd = [nvcc, *ARCH, *FLAGS, *per_file, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            print(r.stdout + r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
