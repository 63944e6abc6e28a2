"""Build the CUDA library ``_lib/liblbpf.so`` for sm_103a (GB300).

Each storage type's kernels live in their own translation unit, compiled in
parallel with nvcc, then linked with the host runtime into one shared library
with a plain C ABI (``include/lbpf.h``).  Usage: ``python -m
paper_1602_07483_gb300.build`` or ``build()`` from Python.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_lib")
LIB = os.path.join(OUT_DIR, "liblbpf.so")
SOURCES = ["lbpf_api.cu", "kern_f64.cu", "kern_f32.cu", "kern_f16.cu", "kern_bf16.cu", "kern_tile_f32.cu",
           "kern_f32_b8.cu", "kern_step_f32.cu", "kern_step_f16.cu", "kern_step_bf16.cu",
           "kern_node_f64.cu", "kern_node_f32.cu", "kern_node_f16.cu", "kern_node_bf16.cu",
           "kern_moment_f64.cu", "kern_moment_f32.cu", "kern_moment_f16.cu", "kern_moment_bf16.cu",
           "kern_pair_f32.cu", "kern_pair_f16.cu", "kern_pair_bf16.cu",
           "lbpf_noalloc.cu"]
HEADERS = ["lbpf_lattice.cuh", "lbpf_node.cuh", "lbpf_dev.cuh", "lbpf_nodewise.cuh", "lbpf_nodepair.cuh", "lbpf_plane.cuh", "lbpf_aux.cuh", "lbpf_table.h", "lbpf_table_impl.cuh", "lbpf_plan.h"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    """Compile (if stale) and link the library; return its path."""
    os.makedirs(os.path.join(OUT_DIR, "obj"), exist_ok=True)
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(HERE, "..", "include", "lbpf.h")]
    cc = nvcc()
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OUT_DIR, "obj", src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + hdrs):
            cmd = [cc] + ARCH + FLAGS + ["-c", s, "-o", o]
            if ptxas_info:
                cmd += ["-Xptxas", "-v"]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    workers = max(1, min(len(jobs), os.cpu_count() or 1))
    failed = []
    if jobs:
        with cf.ThreadPoolExecutor(workers) as ex:
            for cmd, r in ex.map(run, jobs):
                if verbose or ptxas_info or r.returncode:
                    sys.stderr.write(r.stdout + r.stderr)
                if r.returncode:
                    failed.append(" ".join(cmd))
    if failed:
        raise RuntimeError("nvcc failed:\n" + "\n".join(failed))
    if force or _stale(LIB, objs):
        tmp = LIB + ".%d.tmp" % os.getpid()
        cmd = [cc] + ARCH + ["-shared", "-o", tmp] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode:
            raise RuntimeError("link failed: %s\n%s" % (" ".join(cmd), r.stdout + r.stderr))
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
