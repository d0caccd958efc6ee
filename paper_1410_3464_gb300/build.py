"""Build the CUDA library in-tree: one nvcc process per translation unit (in
parallel), linked into paper_1410_3464_gb300/_lib/libpslbm.so for sm_103a."""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_lib")
LIB = os.path.join(OUT_DIR, "libpslbm.so")
SOURCES = ["kernels_f64.cu", "kernels_f32.cu", "kernels_f32h.cu", "kernels_f32b.cu", "runtime.cu", "noalloc.cu", "serve.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# No product is fused into a sum but where the source says so: otherwise the compiler
# may do it in one instantiation of the FP64 kernels (one simulation, batch of like or
# unlike members, VOP and amendment in one launch or two) and not in another, and
# their bits would differ.  The FP32 units keep the default, on which the bits of
# their expf and expm1f rest.
FLAGS = {"kernels_f64.cu": ["-fmad=false"]}


def nvcc():
    exe = shutil.which("nvcc")
    if exe:
        return exe
    cand = "/usr/local/cuda/bin/nvcc"
    if os.path.exists(cand):
        return cand
    raise RuntimeError("nvcc not found")


def compile_command(src, cc="nvcc"):
    obj = os.path.join(OUT_DIR, "obj", src.replace(".cu", ".o"))
    return ([cc] + ARCH + ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC"] + FLAGS.get(src, []) +
            ["-c", os.path.join(CSRC, src), "-o", obj])


def _stale(obj, src_files):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(s) > t for s in src_files)


def build(verbose=False, force=False):
    os.makedirs(os.path.join(OUT_DIR, "obj"), exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers += [os.path.join(os.path.dirname(HERE), "include", "pslbm.h"), os.path.abspath(__file__)]
    cc = nvcc()
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OUT_DIR, "obj", src.replace(".cu", ".o"))
        if force or _stale(o, [s] + headers):
            jobs.append((src, compile_command(src, cc)))
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
            futs = {ex.submit(subprocess.run, cmd, capture_output=True, text=True): src for src, cmd in jobs}
            for f in cf.as_completed(futs):
                r = f.result()
                if r.returncode != 0:
                    raise RuntimeError(f"nvcc failed on {futs[f]}:\n{r.stderr[-4000:]}")
                if verbose and r.stderr:
                    print(r.stderr, file=sys.stderr)
    objs = [os.path.join(OUT_DIR, "obj", s.replace(".cu", ".o")) for s in SOURCES]
    if force or jobs or not os.path.exists(LIB):
        cmd = [cc] + ARCH + ["-shared", "-o", LIB] + objs + ["-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stderr[-4000:]}")
    return LIB


if __name__ == "__main__":
    print(build(verbose=True, force="--force" in sys.argv))
