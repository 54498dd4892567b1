"""Build libhom.so (sm_103a) in-tree with nvcc.

Each .cu translation unit is compiled in parallel, then linked into
paper_2110_00733_gb300/lib/libhom.so.  Nothing here falls back to another
architecture or to the CPU.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "lib")
LIB = os.path.join(OUT_DIR, "libhom.so")
SOURCES = ["hom_kernels_f32.cu", "hom_kernels_f64.cu", "hom_x1l_a.cu", "hom_x1l_b.cu", "hom_x1l_c.cu",
           "hom_f64_x1_a.cu", "hom_f64_x1_b.cu", "hom_f64_x1_c.cu", "hom_f64_x1l_a.cu", "hom_f64_x1l_b.cu", "hom_f64_x1l_c.cu",
           "hom_f64_x2_a.cu", "hom_f64_x2_b.cu", "hom_f64_x2_c.cu", "hom_f64_x3_a.cu", "hom_f64_x3_b.cu", "hom_f64_x3_c.cu",
           "hom_f64_ord_a.cu", "hom_f64_ord_b.cu",
           "hom_x2_a.cu", "hom_x2_b.cu", "hom_x2_c.cu", "hom_x3_a.cu", "hom_x3_b.cu", "hom_x3_c.cu", "hom_common.cu", "hom_api.cu", "hom_noalloc.cu",
           "hom_batch.cu", "hom_cg.cu", "hom_pfs.cu", "hom_j2.cu", "net.cu", "net_tc.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    for f in os.listdir(CSRC):
        if os.path.getmtime(os.path.join(CSRC, f)) > t:
            return True
    for name in ("hom.h", "hom_net.h"):
        hdr = os.path.join(os.path.dirname(HERE), "include", name)
        if os.path.exists(hdr) and os.path.getmtime(hdr) > t:
            return True
    return False


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(os.path.join(OUT_DIR, "obj"), exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(OUT_DIR, "obj", src.replace(".cu", ".o"))
        cmd = [nvcc, *ARCH, *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.append("-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    with ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", *objs, "-o", tmp, "-lcudart", "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
