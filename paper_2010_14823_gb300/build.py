"""Build the CUDA library (sm_103a) in-tree with nvcc."""
from __future__ import annotations

import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(HERE, "libcasim.so")
# the same library with every index checked (-DCASIM_DEBUG): an index outside
# its array sets CASIM_EFLAG_INDEX in the error word and the access is skipped
LIB_DEBUG = os.path.join(HERE, "libcasim_debug.so")
# the C ABI with the batch and network kernels, and the step kernels by configuration
SOURCES = [os.path.join(CSRC, f) for f in ("casim.cu", "casim_step_cold.cu", "casim_step_aero.cu", "casim_step_tri.cu",
                                           "casim_step_warm.cu", "casim_step_warm_ext.cu")]
DEPS = SOURCES + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))] + [
    os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE) if f.endswith(".h")]
# instruction-throughput probes (measurement support, its own library)
PEAKS_LIB = os.path.join(HERE, "libcasim_peaks.so")
PEAKS_SOURCES = [os.path.join(CSRC, "casim_peaks.cu")]
PEAKS_DEPS = PEAKS_SOURCES + [os.path.join(INCLUDE, "casim_peaks.h")]

# -ftz=true: FP32 arithmetic flushes subnormal values to zero.  The mixed
# step's FP32 values are normal or zero by construction (its FP64 -> FP32
# conversion flushes magnitudes below 2^-126), so its results are unchanged,
# bit for bit, while FP32 divisions and the like skip their subnormal handling
# (measured: 2.13 -> 2.02 ms per 512x512x150 step).  FP64 code is unaffected.
NVCC_FLAGS = ["-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-lineinfo", "-std=c++17", "-ftz=true",
              "-Xcompiler", "-fPIC", "-I" + INCLUDE]
LINK_FLAGS = ["-shared", "-ldl"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(lib: str, deps: list[str]) -> bool:
    return not os.path.exists(lib) or os.path.getmtime(lib) < max(os.path.getmtime(p) for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile libcasim.so, its index-checked build libcasim_debug.so and
    libcasim_peaks.so where missing or older than their sources: every
    translation unit of each at once, then the links."""
    jobs = []
    for lib, srcs, deps, extra in ((LIB, SOURCES, DEPS, []), (LIB_DEBUG, SOURCES, DEPS, ["-DCASIM_DEBUG"]),
                                   (PEAKS_LIB, PEAKS_SOURCES, PEAKS_DEPS, [])):
        if force or _stale(lib, deps):
            objs = [f"{lib}.{os.path.basename(s)}.o" for s in srcs]
            more = extra + (["-Xptxas", "-v"] if verbose else [])
            jobs.append((lib, objs, [subprocess.Popen([nvcc()] + NVCC_FLAGS + more + ["-c", "-o", o, s])
                                     for s, o in zip(srcs, objs)]))
    for lib, objs, procs in jobs:
        for p in procs:
            if p.wait() != 0:
                raise subprocess.CalledProcessError(p.returncode, "nvcc " + os.path.basename(lib))
        subprocess.run([nvcc()] + NVCC_FLAGS[:2] + LINK_FLAGS + ["-o", lib + ".tmp"] + objs, check=True)
        for o in objs:
            os.remove(o)
        os.replace(lib + ".tmp", lib)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose=True)
