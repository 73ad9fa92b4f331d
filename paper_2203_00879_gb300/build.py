"""Builds libnopcs.so in-tree with nvcc for sm_103a (no CMake, no torch)."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libnopcs.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]
# per-file nvcc flags (none at present)
PER_FILE_FLAGS = {}


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale(out, deps):
    if not os.path.exists(out):
        return True
    t = os.path.getmtime(out)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    os.makedirs(OBJ, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    headers.append(os.path.join(HERE, "..", "include", "nopcs.h"))
    srcs = sources()
    objs = [os.path.join(OBJ, os.path.basename(s)[:-3] + ".o") for s in srcs]

    def compile_one(pair):
        src, obj = pair
        if not force and not _stale(obj, [src] + headers):
            return ""
        cmd = [NVCC, *ARCH, *FLAGS, *PER_FILE_FLAGS.get(os.path.basename(src), []), *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
        return r.stdout + r.stderr

    with ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        logs = list(ex.map(compile_one, zip(srcs, objs)))
    if verbose:
        for lg in logs:
            if lg:
                sys.stdout.write(lg)
    if force or _stale(LIB, objs):
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [NVCC, *ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", tmp, *objs]
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True,
          extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else [])
    print(LIB)


# Sources of each kernel kind of the mixed form (the profiler counters kept are of
# that form).  The filter runs the FP32 sweeps or, for coefficients near 1/2, the
# sub-domain sweep, and then its update.
_LINE = ["line_kernels.cu", "line_body.cuh", "line_solve.cuh"]
_SWEEP = ["sweep32.cuh", "sweep32_kernels.cu"]
KERNEL_FILES = {
    "prep": ["rk_kernels.cu", "fp_bits.cuh"], "wall_bc": ["rk_kernels.cu", "wall_body.cuh", "fp_bits.cuh"],
    "diagnostics": ["rk_kernels.cu", "fp_bits.cuh"],
    "sweep_x": _SWEEP, "sweep_y": _SWEEP, "sweep_z": _SWEEP,
    "filter": _SWEEP + _LINE + ["rk_kernels.cu", "fp_bits.cuh"],
    "visc_rk_update": ["visc_kernel.cu", "visc_body.cuh", "fp_bits.cuh"],
}


def source_hash(files=None) -> str:
    """Content hash of CUDA sources (all of them, or the named files plus the
    internal header); tags profiler counters with the code they measured."""
    import hashlib
    h = hashlib.sha256()
    names = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
    if files is not None:
        names = sorted(set(files) | {"nopcs_internal.cuh"})
    for f in names:
        with open(os.path.join(CSRC, f), "rb") as fh:
            h.update(f.encode() + b"\0" + fh.read())
    return h.hexdigest()[:16]
