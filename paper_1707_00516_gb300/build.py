"""Build the CUDA library in place for sm_103a (GB300).

Each ``csrc/*.cu`` compiles to an object under ``_build/`` in parallel; the
objects link into ``libfastid.so`` next to this file.  The public header is
``include/fastid.h`` at the repository root.

``build_peaks()`` compiles the roofline microbenchmarks (``probe/peaks.cu``)
into ``libfastid_peaks.so``; the comparison library does not link them.

``build(debug=True)`` makes ``libfastid_debug.so`` (objects under
``_build_debug/``) with FASTID_DEBUG defined: device-side consistency checks
that record ST_DEVICE in the context's status word instead of trusting the
schedule, and a host-side self-check of every tensor schedule.  Load it with
``binding.load_library(build.LIB_DEBUG)``.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libfastid.so")
BUILD_DEBUG = os.path.join(PKG, "_build_debug")
LIB_DEBUG = os.path.join(PKG, "libfastid_debug.so")
PEAKS_SRC = os.path.join(PKG, "probe", "peaks.cu")
LIB_PEAKS = os.path.join(PKG, "libfastid_peaks.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
              "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def headers() -> list[str]:
    """Every header a source may include: a change of one rebuilds all objects,
    which share its structures."""
    return sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) +
                  glob.glob(os.path.join(INCLUDE, "*.h")))


def _deps() -> list[str]:
    return sources() + headers() + [__file__]


def _stale(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra_flags: list[str] | None = None,
          debug: bool = False) -> str:
    """Compile (if stale) and return the path of libfastid.so (libfastid_debug.so
    with debug=True)."""
    lib_path, build_dir = (LIB_DEBUG, BUILD_DEBUG) if debug else (LIB, BUILD)
    deps = _deps()
    if not force and not _stale(lib_path, deps):
        return lib_path
    os.makedirs(build_dir, exist_ok=True)
    nvcc = _nvcc()
    extra = list(extra_flags or []) + (["-DFASTID_DEBUG"] if debug else [])

    def compile_one(src: str) -> str:
        obj = os.path.join(build_dir, os.path.basename(src)[:-3] + ".o")
        if force or _stale(obj, [src, __file__] + headers()):
            cmd = [nvcc, *ARCH, *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
            if verbose:
                print(" ".join(cmd), file=sys.stderr)
            r = subprocess.run(cmd, capture_output=True, text=True)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
            if verbose and r.stderr:
                print(r.stderr, file=sys.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=max(1, min(8, os.cpu_count() or 1))) as ex:
        objs = list(ex.map(compile_one, sources()))
    tmp = lib_path + f".tmp{os.getpid()}"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, lib_path)
    return lib_path


def build_peaks(force: bool = False) -> str:
    """Compile (if stale) and return the path of libfastid_peaks.so."""
    if not force and not _stale(LIB_PEAKS, [PEAKS_SRC, __file__]):
        return LIB_PEAKS
    tmp = LIB_PEAKS + f".tmp{os.getpid()}"
    cmd = [_nvcc(), *ARCH, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", PEAKS_SRC, "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {PEAKS_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB_PEAKS)
    return LIB_PEAKS


if __name__ == "__main__":
    # python -m paper_1707_00516_gb300.build [--force] [-v] [--debug]
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
