"""Build the in-tree CUDA library for sm_103a (nvcc only; no cmake).

    python -m paper_1306_6445_gb300._build        # or __graft_entry__.build()

Translation units are compiled in parallel into ``_build/`` and linked into
``_lib/liblb_gb300.so`` next to this file. A source newer than the library
triggers a rebuild; ``force=True`` always rebuilds.
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
LIBDIR = os.path.join(HERE, "_lib")
LIB = os.path.join(LIBDIR, "liblb_gb300.so")
SOURCES = ["lb_step_f32.cu", "lb_step_f32_stage.cu", "lb_step_f64.cu", "lb_step_f64_stage.cu",
           "lb_step_bf16.cu", "lb_step_bf16_stage.cu", "lb_batch_kernels.cu", "lb_batch_stage.cu",
           "lb_tile_f32.cu", "lb_tile_bf16.cu",
           "lb_split_f64.cu", "lb_batch_tile.cu", "lb_cluster.cu", "lb_resident.cu", "lb_kernels.cu", "lb_api.cu", "lb_thermo.cpp", "lb_noalloc.cu", "lb_batch.cu",
           "lb_mlp.cu", "lb_probe.cu"]
HEADERS = ["lb_internal.h", "lb_device.cuh", "lb_step.cuh", "lb_tile.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "--expt-relaxed-constexpr",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-O2", "-Xptxas", "-v"] + ARCH


def nvcc() -> str:
    cand = [os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"]
    for c in cand:
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build the library")


def _deps():
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS]
    deps += [os.path.join(ROOT, "include", h) for h in ("lb.h", "lb_mlp.h")]
    return deps


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(d) <= t for d in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    exe = nvcc()

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
        cmd = [exe] + NVCC_FLAGS + ["-I", os.path.join(ROOT, "include"), "-c",
                                    os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    if verbose:
        for _, log in results:
            sys.stderr.write(log)
    with open(os.path.join(BUILD, "ptxas.log"), "w") as fh:
        for _, log in results:
            fh.write(log)
    tmp = LIB + ".tmp"
    cmd = [exe, "-shared"] + ARCH + ["-o", tmp] + [o for o, _ in results]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
