"""Build the CUDA library liblbm.so in-tree with nvcc for sm_103a.

Translation units are compiled in parallel and linked into
``paper_1710_09472_gb300/_build/liblbm.so``; the Python binding loads that
file and nothing else.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "liblbm.so")
SOURCES = ["lbm_step_f16_x.cu", "lbm_step_bf16_x.cu", "lbm_step_f16.cu", "lbm_step_bf16.cu", "lbm_step_f16_x_n.cu",
           "lbm_step_bf16_x_n.cu", "lbm_step_f16_n.cu", "lbm_step_bf16_n.cu", "lbm_step_f32.cu", "lbm_step_f32_x.cu",
           "lbm_api.cu", "lbm_kernels.cu", "lbm_adjoint.cu", "lbm_static.cu", "lbm_adjoint_f32.cu",
           "lbm_adjoint_f16.cu", "lbm_adjoint_bf16.cu", "lbm_adjoint_f32_x.cu", "lbm_adjoint_f16_x.cu",
           "lbm_adjoint_bf16_x.cu", "lbm_adjoint_f32_lmu.cu", "lbm_adjoint_f16_lmu.cu", "lbm_adjoint_bf16_lmu.cu",
           "lbm_multi_f32.cu", "lbm_multi_f16.cu", "lbm_multi_bf16.cu", "lbm_thermal.cu", "lbm_fd.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build liblbm")
    return path


def _flags(extra=()):
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                   "-I", os.path.join(ROOT, "include"), "-I", CSRC, *extra]


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    os.makedirs(BUILD, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    headers.append(os.path.join(ROOT, "include", "lbm.h"))
    objs = []
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            jobs.append([nvcc(), *_flags(extra_flags), "-c", s, "-o", o])
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
            results = list(ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs))
        for cmd, r in zip(jobs, results):
            if verbose or r.returncode != 0:
                print(" ".join(cmd))
                print(r.stdout, r.stderr)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed for {cmd[-3]}")
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            print(r.stdout, r.stderr)
            raise RuntimeError("link of liblbm.so failed")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose=True))
