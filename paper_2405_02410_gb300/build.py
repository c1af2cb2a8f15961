"""Build libpss.so (the sm_103a kernels and the C ABI of include/pss.h) in-tree.

nvcc compiles the translation units in parallel (one -gencode, sm_103a)
and links them into paper_2405_02410_gb300/_lib/libpss.so.
"""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIBDIR = os.path.join(HERE, "_lib")
LIB = os.path.join(LIBDIR, "libpss.so")
SOURCES = ["pss_api.cu", "pss_kern_f32.cu", "pss_kern_f64.cu", "pss_kern_f32_r16.cu", "pss_kern_f64_r16.cu", "pss_kern_f64_r4.cu", "pss_kern_f64_r2.cu",
           "pss_kern_fast2d.cu", "pss_kern_persist.cu", "pss_kern_persist_kpz.cu", "pss_kern_persist_adj.cu",
           "pss_kern_line_f32.cu", "pss_kern_line_f64.cu", "pss_kern_terms_f32.cu", "pss_kern_regs.cu",
           *[f"pss_kern_res2d_{n}.cu" for n in (32, 64, 128, 256, 512)]]
HEADERS = ["pss_device.cuh", "pss_internal.h", "pss_kernels.cuh", "pss_fast2d.cuh", "pss_persist2d.cuh", "pss_adj2d.cuh", "pss_persist_adj.cuh",
           "pss_resident2d.cuh", "pss_line.cuh", "pss_terms.cuh", "pss_regs.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-fno-strict-aliasing",
              "--expt-relaxed-constexpr"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _inputs():
    files = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    files.append(os.path.join(os.path.dirname(HERE), "include", "pss.h"))
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(LIBDIR, exist_ok=True)
    nv = nvcc()
    objs = []
    cmds = []
    for src in SOURCES:
        obj = os.path.join(LIBDIR, src.replace(".cu", ".o"))
        objs.append(obj)
        cmds.append([nv, *ARCH, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose:
            sys.stdout.write(r.stdout + r.stderr)

    with concurrent.futures.ThreadPoolExecutor(len(cmds)) as ex:
        list(ex.map(run, cmds))
    tmp = LIB + f".{os.getpid()}.tmp"
    run([nv, *ARCH, "-shared", "-o", tmp, *objs])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
