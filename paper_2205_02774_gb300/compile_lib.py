"""Build libstglbm.so (CUDA for sm_103a) in-tree with nvcc.

Each translation unit is compiled in parallel, then linked into one shared
library next to this file.  Only one -gencode is emitted (sm_103a).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libstglbm.so")
STEP_TUS = ["step_f32_reg.cu", "step_f32_bgk.cu", "step_f16_reg.cu", "step_f16_reg_quad.cu",
            "step_f16_bgk.cu", "step_f16_bgk_quad.cu", "step_f16sr_reg.cu", "step_f16sr_reg_quad.cu", "step_f16sr_bgk.cu",
            "step_f16sr_bgk_quad.cu", "step_f32_reg_row.cu", "step_f32_bgk_row.cu", "step_f16_reg_row.cu",
            "step_f16_bgk_row.cu", "step_f16sr_reg_row.cu", "step_f16sr_bgk_row.cu"]
SOURCES = ["capi.cu", "step_kernel.cu", *STEP_TUS, "inlet_kernel.cu", "noalloc.cu", "batch.cu", "serve.cu", "probe.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", CSRC, "-I", INCLUDE,
              "--expt-relaxed-constexpr"]
# The FP32 step arithmetic uses the hardware approximate reciprocal and square
# root (a few ulp, far inside the parity tolerance) and flushes denormals; the
# FP64 setup code is unaffected by these flags.
FAST_FP32 = ["-ftz=true", "-prec-div=false", "-prec-sqrt=false"]
FAST_TUS = {"step_kernel.cu", *STEP_TUS}


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "stg_lbm.h"))
    files.append(os.path.abspath(__file__))
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        fast = FAST_FP32 if src in FAST_TUS else []
        cmd = [nvcc, *ARCH, *NVCC_FLAGS, *fast, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    if verbose or ptxas_info:
        for _, log in results:
            if log:
                print(log, file=sys.stderr)
    objs = [o for o, _ in results]
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "shared"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
