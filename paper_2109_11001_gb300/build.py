"""Compile the CUDA library ``libkg.so`` in-tree for sm_103a with nvcc.

Each translation unit is compiled in parallel, then linked into one shared
library with the CUDA runtime linked statically (no dependence on the
runtime's location at load time).
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libkg.so")
SOURCES = ["kg_api.cu", "kg_md.cu", "kg_step.cu", "kg_resident.cu", "kg_resident_small.cu", "kg_resident_tiled.cu", "kg_db.cu", "kg_obs.cu", "kg_learned.cu", "kg_mlp.cu", "kg_ppa.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# the mixed path's step kernels: binary32 denormals flushed to zero and the
# approximate divide and square root (its arithmetic never meets a denormal;
# the rounding changes stay far inside the parity bars)
STEP_FLAGS = ["-ftz=true", "-prec-div=false", "-prec-sqrt=false"]
PER_FILE = {"kg_step.cu": STEP_FLAGS, "kg_resident.cu": STEP_FLAGS, "kg_resident_small.cu": STEP_FLAGS,
            "kg_resident_tiled.cu": STEP_FLAGS}
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale() -> bool:
    if not os.path.exists(OUT):
        return True
    t = os.path.getmtime(OUT)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "kg.h"), __file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    if not force and not _stale():
        return OUT
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    procs, objs = [], []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc(), *ARCH, *FLAGS, *PER_FILE.get(src, []), *extra, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    errors = []
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            (errors if p.returncode else []).append(f"--- {src}\n{out.decode(errors='replace')}")
            if verbose:
                print(out.decode(errors="replace"), file=sys.stderr)
    if errors:
        raise RuntimeError("nvcc failed:\n" + "\n".join(errors))
    tmp = OUT + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc(), *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs])
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv,
          extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else ())
    print(OUT)
