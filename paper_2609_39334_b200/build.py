"""Builds the CUDA library (libspecscale.so) in-tree with nvcc for sm_100a.

    python -m paper_2609_39334_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libspecscale.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
         "-Xcompiler", "-fPIC"]
# Per-file additions: ptxas's most register-conserving setting schedules the softmax loop of the default tile kernel
# slightly better (measured); a less conserving one than usual suits the exponentials of the sampler (922 rows of 151936:
# 184.3 us at the default of 5, 181.8 at 3, 188.4 at 7 and 10).
FILE_FLAGS = {"attn_umma_split.cu": ["-Xptxas", "--register-usage-level=10"],
              "branch_sample.cu": ["-Xptxas", "--register-usage-level=3"]}


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(_HERE, "..", "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def build(force: bool = False, verbose: bool = False, defines=(), suffix: str = "") -> str:
    """Builds libspecscale<suffix>.so.  `defines` are extra -D macros (an instrumented or checked variant gets its own
    suffix and object directory); SS_NVCC_DEFINES in the environment adds more, comma separated."""
    defines = list(defines) + [d for d in os.environ.get("SS_NVCC_DEFINES", "").split(",") if d]
    lib = LIB[:-3] + suffix + ".so"
    if not force and not _stale(lib):
        return lib
    objdir = os.path.join(_HERE, "build" + suffix)
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [NVCC, *FLAGS, *[f"-D{d}" for d in defines], *FILE_FLAGS.get(os.path.basename(src), []), "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)} ---\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = lib + f".tmp{os.getpid()}"
    subprocess.check_call([NVCC, "-shared", "-o", tmp, *objs, "-Xcompiler", "-fPIC"])
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
