"""Build libpathmc.so in-tree with nvcc for sm_103a.

Each CUDA translation unit is compiled in parallel, then linked into
``paper_1811_04156_gb300/_build/libpathmc.so``.  The benchmark harness's
pipe-rate microbenchmark (csrc/probe/) is a library of its own,
``_build/libpmcprobe.so``, outside the product library.  Rebuilds only when
a source or header is newer than the library.
"""
from __future__ import annotations

import concurrent.futures as cf
import fcntl
import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libpathmc.so")
PROBE_SRC = os.path.join(CSRC, "probe", "pipe_rates.cu")
PROBE_LIB = os.path.join(BUILD, "libpmcprobe.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
              "-I", INCLUDE] + ARCH


# The chain kernels are built twice: as they are, and with subnormals flushed,
# for scenes in which no subnormal can arise (flush_is_exact in pmc_capi.cu);
# their approximate logarithms, roots and divisions otherwise rescale subnormal
# arguments, two to three instructions for each of the 20 to 30 per proposal.
FLUSH_SOURCES = ("pmc_chain.cu", "pmc_group.cu", "pmc_lane.cu")
FLUSH_FLAGS = ["-ftz=true", "-DPMC_FLUSH_SUBNORMALS"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpathmc")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    """What the library is made from, this file with its flags included."""
    return [os.path.abspath(__file__)] + _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(INCLUDE, "*.h"))


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in _deps())


def _build_probe(nvcc: str) -> None:
    if os.path.exists(PROBE_LIB) and all(os.path.getmtime(PROBE_LIB) >= os.path.getmtime(p)
                                         for p in (PROBE_SRC, os.path.abspath(__file__))):
        return
    tmp = PROBE_LIB + f".tmp{os.getpid()}"
    r = subprocess.run([nvcc, "-shared", "-o", tmp, PROBE_SRC] + NVCC_FLAGS, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {PROBE_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, PROBE_LIB)


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    """Build the library (and the probe library) if a source is newer.  Processes
    that build at once (ranks of a multi-process test) take turns on a lock
    file in the build folder, so that none links another's half-written
    objects; whoever comes second finds the library up to date."""
    os.makedirs(BUILD, exist_ok=True)
    with open(os.path.join(BUILD, ".lock"), "w") as lock:
        fcntl.flock(lock, fcntl.LOCK_EX)
        try:
            return _build_locked(force, verbose, ptxas_info)
        finally:
            fcntl.flock(lock, fcntl.LOCK_UN)


def _build_locked(force: bool, verbose: bool, ptxas_info: bool) -> str:
    if force and os.path.exists(PROBE_LIB):
        os.unlink(PROBE_LIB)
    _build_probe(_nvcc())
    if not force and up_to_date():
        return LIB
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if ptxas_info else []

    units = [(src, "", []) for src in _sources()]
    units += [(src, ".flush", FLUSH_FLAGS) for src in _sources() if os.path.basename(src) in FLUSH_SOURCES]

    def compile_one(unit):
        src, variant, flags = unit
        obj = os.path.join(BUILD, os.path.basename(src) + variant + ".o")
        cmd = [nvcc, "-c", src, "-o", obj] + NVCC_FLAGS + flags + extra
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        results = list(ex.map(compile_one, units))
    if verbose or ptxas_info:
        for _, log in results:
            if log:
                sys.stderr.write(log)
    objs = [o for o, _ in results]
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-shared", "-o", tmp] + objs + ARCH
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
