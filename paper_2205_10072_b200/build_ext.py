"""Compiles the CUDA sources of this package for sm_100a into libbcs.so (in-tree, next to this file)."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
LIB_PATH = os.path.join(_PKG, "libbcs.so")
SOURCES = sorted(glob.glob(os.path.join(_PKG, "csrc", "*.cu")))
HEADERS = sorted(glob.glob(os.path.join(_ROOT, "include", "*.h")) +
                 glob.glob(os.path.join(_PKG, "csrc", "*.cuh")))
# The unit with the kernels that read the constants below: all of them, so that these are in the library once (loaded by the first
# call), and without line information, with which nvcc adds the unit's PTX, 7 MB of it the constants as text.  (First calls of a
# process, one p and a batch: 5.5 + 0.2 ms, of which some 2 MB of quad_kernel for each q take 1; before that kernel 4.4 + 0.2, with line information 7.7 + 0.2,
# in two such units 7.2 + 4.3, the file 8.2 (before that kernel 5.8), 13.8, 23 MB.)
ROWS_UNIT = os.path.join(_PKG, "csrc", "rows.cu")
# The packed rows of all shapes of segments, written by a small program at build time.
ROW_TABLE = os.path.join(_PKG, "csrc", "row_table.inc")
ROW_TABLE_SOURCE = os.path.join(_PKG, "csrc", "gen", "row_table.c")
# The calls of the library for Python (csrc/calls.c), linked to it.
CALLS_PATH = os.path.join(_PKG, "_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
CALLS_SOURCE = os.path.join(_PKG, "csrc", "calls.c")
# The benchmark's integer-rate probe is a library of its own: it is not part of the product and
# only bench.py loads it.
PROBE_LIB_PATH = os.path.join(_PKG, "libbcs_probe.so")
PROBE_SOURCES = sorted(glob.glob(os.path.join(_PKG, "csrc", "probe", "*.cu")))
PROBE_HEADERS = sorted(glob.glob(os.path.join(_PKG, "csrc", "probe", "*.h")))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    "--shared", "-Xcompiler", "-fPIC",
    "-I", os.path.join(_ROOT, "include"),
]


def _stale(lib: str, deps: list) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(f) > t for f in deps)


def stale() -> bool:
    return _stale(LIB_PATH, SOURCES + HEADERS + [ROW_TABLE_SOURCE])


def _nvcc(lib: str, sources: list, verbose: bool, extra: list = ()) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = lib + ".%d.tmp" % os.getpid()
    says = ["-Xptxas", "-v"] if verbose else []
    sources, unit = list(sources), tmp + ".o"
    try:
        if ROWS_UNIT in sources:
            flags = [f for f in NVCC_FLAGS if f not in ("--shared", "-lineinfo")]
            subprocess.check_call([nvcc] + flags + says + ["-c", "-o", unit, ROWS_UNIT])
            sources[sources.index(ROWS_UNIT)] = unit
        subprocess.check_call([nvcc] + NVCC_FLAGS + ["-Xlinker", "-soname=" + os.path.basename(lib)] + list(extra) + says + ["-o", tmp] + sources)
    finally:
        if os.path.exists(unit):
            os.remove(unit)
    os.replace(tmp, lib)


def build_row_table(force: bool = False) -> str:
    """Compiles and runs csrc/gen/row_table.c, which writes the constants that the row kernels include."""
    if force or _stale(ROW_TABLE, [ROW_TABLE_SOURCE]):
        tmp = ROW_TABLE + ".%d.tmp" % os.getpid()
        exe = tmp + ".exe"
        try:
            subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-o", exe, ROW_TABLE_SOURCE])
            with open(tmp, "wb") as out:
                subprocess.check_call([exe], stdout=out)
            os.replace(tmp, ROW_TABLE)
        finally:
            for left in (exe, tmp):
                if os.path.exists(left):
                    os.remove(left)
    return ROW_TABLE


def build(force: bool = False, verbose: bool = False) -> str:
    """Runs nvcc (cross-compiles without a GPU).  Returns the path of the shared library."""
    build_row_table(force)
    if force or stale():
        _nvcc(LIB_PATH, SOURCES, verbose)
    build_calls(force)
    return LIB_PATH


def build_calls(force: bool = False) -> str:
    """The extension module with the library's calls (without Python's headers: none, ctypes serves)."""
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")):
        return ""
    if force or _stale(CALLS_PATH, [CALLS_SOURCE, LIB_PATH] + HEADERS):
        tmp = CALLS_PATH + ".%d.tmp" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC",
                               "-I", include, "-I", os.path.join(_ROOT, "include"),
                               "-o", tmp, CALLS_SOURCE, LIB_PATH, "-Wl,-rpath,$ORIGIN"])
        os.replace(tmp, CALLS_PATH)
    return CALLS_PATH


def build_probe(force: bool = False, verbose: bool = False) -> str:
    """The benchmark's probe library (bcs_probe_int_rate), separate from libbcs.so."""
    if force or _stale(PROBE_LIB_PATH, PROBE_SOURCES + PROBE_HEADERS + HEADERS):
        _nvcc(PROBE_LIB_PATH, PROBE_SOURCES, verbose, ["-I", os.path.join(_PKG, "csrc")])
    return PROBE_LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
    print(build_probe(force=True, verbose=True))
