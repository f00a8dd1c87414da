"""Build the CUDA library libp3dfft_gb300.so in-tree for sm_103a.

nvcc compiles each translation unit in parallel, then links one shared
library with the CUDA runtime linked statically, so the binding needs nothing
but the driver at load time.
"""
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(OUT_DIR, "libp3dfft_gb300.so")
SOURCES = ["p3_plan.cu", "p3_kernels.cu", "p3_pow2.cu", "p3_pow2_f32.cu", "p3_pow2_f64.cu", "p3_noalloc.cu", "p3_tc.cu",
           "p3_fused.cu", "p3_batch.cu", "p3_fix64.cu", "p3_fix64_cc.cu", "p3_fix64_cs.cu",
           "p3_fix64_ecc.cu", "p3_fix64_ecs.cu", "p3_fix64_row.cu", "p3_fix64_pair.cu", "p3_line32.cu",
           "p3_line32_a.cu", "p3_line32_b.cu"]
HEADERS = [os.path.join(CSRC, "p3_internal.h"), os.path.join(CSRC, "p3_dft.cuh"), os.path.join(CSRC, "p3_pow2.cuh"),
           os.path.join(CSRC, "p3_fix64.cuh"), os.path.join(CSRC, "p3_line32.cuh"), os.path.join(CSRC, "p3_launch.cuh"), os.path.join(CSRC, "p3_copy.cuh"), os.path.join(ROOT, "include", "p3dfft_gb300.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    os.makedirs(OUT_DIR, exist_ok=True)
    nvcc = _nvcc()
    objs, jobs = [], []
    for src in SOURCES:
        path = os.path.join(CSRC, src)
        obj = os.path.join(OUT_DIR, src.replace(".cu", ".o"))
        objs.append(obj)
        if force or _stale(obj, [path] + HEADERS):
            cmd = [nvcc] + ARCH + FLAGS + list(extra) + ["-c", path, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n%s\n%s" % (" ".join(cmd), r.stderr))
        if verbose and r.stderr:
            print(r.stderr, flush=True)

    with ThreadPoolExecutor(max_workers=max(1, len(jobs))) as ex:
        list(ex.map(run, jobs))
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        run([nvcc] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv,
                extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else ()))
