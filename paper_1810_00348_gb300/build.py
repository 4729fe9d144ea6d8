"""Build libkgs.so (the C-ABI solver library) in-tree for GB300 (sm_103a).

    python -m paper_1810_00348_gb300.build [--force] [--verbose-ptxas]

Each CUDA translation unit is compiled in parallel with nvcc, then linked into
paper_1810_00348_gb300/libkgs.so.  No torch headers or types are involved.
"""
import argparse
import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkgs.so")
BUILD = os.path.join(HERE, "_build")
SOURCES = ["kgs_runtime.cu", "kgs_tables.cu", "kgs_sweep.cu", "kgs_sweep_f2.cu", "kgs_sweep_d.cu", "kgs_closure.cu", "kgs_noalloc.cu", "kgs_batch.cu", "kgs_autotune.cu", "kgs_nn.cu", "kgs_conv_tc.cu", "kgs_solve.cu"]
HEADERS = [os.path.join(CSRC, "kgs_sweep_dev.cuh"), os.path.join(CSRC, "kgs_internal.h"), os.path.join(CSRC, "kgs_nn.h"), os.path.join(CSRC, "kgs_tables.h"), os.path.join(CSRC, "kgs_ctx.h"), os.path.join(CSRC, "kgs_switch.h"), os.path.join(CSRC, "kgs_pack.h"), os.path.join(ROOT, "include", "kgs.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc():
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _flags(verbose_ptxas=False):
    f = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")] + ARCH
    if verbose_ptxas:
        f += ["-Xptxas", "-v"]
    return f


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose_ptxas: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    flags = _flags(verbose_ptxas)

    def compile_one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        cmd = [nvcc] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    for _, log in results:
        if verbose_ptxas and log:
            sys.stderr.write(log)
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + [o for o, _ in results] + ["-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    ap = argparse.ArgumentParser()
    ap.add_argument("--force", action="store_true")
    ap.add_argument("--verbose-ptxas", action="store_true")
    args = ap.parse_args()
    print(build(force=args.force, verbose_ptxas=args.verbose_ptxas))
