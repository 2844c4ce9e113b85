"""Build libdg.so (the C-ABI library) in-tree with nvcc for sm_103a.

The translation units compile in parallel (the element kernels per number of
points per direction and part) and link into paper_2511_08020_gb300/_lib/libdg.so.  The FP64 throughput probes of the
benchmark (fp64_probe.cu) link into a library of their own,
_lib/libfp64probe.so, so that libdg.so carries only the hot path.  Nothing is
installed elsewhere.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIBDIR = os.path.join(HERE, "_lib")
LIB = os.path.join(LIBDIR, "libdg.so")
SOURCES = ["dg_host.cpp", "dg_kernels.cu", "dg_faces.cu", "dg_moving.cu", "dg_api.cu"]
# one build per number of points per direction (DG_N = N + 1) and part, the slow ones first
ELEMENT_SRC = "dg_element.cu"
ELEMENT_BUILDS = [(n, p) for n in (7, 6, 5, 4, 3, 2) for p in (1, 2, 0)]
PROBE_SRC = "fp64_probe.cu"
PROBE_LIB = os.path.join(LIBDIR, "libfp64probe.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]


def nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found; the library needs the CUDA toolkit to build")
    return path


def _compile(src: str, obj: str, defines: tuple = ()) -> None:
    cmd = [nvcc(), *ARCH, *FLAGS, *defines, "-c", os.path.join(CSRC, src), "-o", obj]
    if src.endswith(".cpp"):
        cmd = [nvcc(), *FLAGS, "-x", "c++", "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"compiling {src} failed:\n{r.stdout}\n{r.stderr}")


def build_probe(force: bool = False) -> str:
    """The benchmark's FP64 throughput probes (libfp64probe.so)."""
    os.makedirs(LIBDIR, exist_ok=True)
    src = os.path.join(CSRC, PROBE_SRC)
    if not force and os.path.exists(PROBE_LIB) and os.path.getmtime(src) <= os.path.getmtime(PROBE_LIB):
        return PROBE_LIB
    tmp = PROBE_LIB + ".tmp"
    cmd = [nvcc(), *ARCH, *FLAGS, "-shared", "-cudart", "shared", "-o", tmp, src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"building libfp64probe.so failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, PROBE_LIB)
    return PROBE_LIB


def dependencies() -> list:
    """Every file libdg.so is made from (sources, headers, this file with its flags and build list)."""
    srcs = [os.path.join(CSRC, s) for s in (*SOURCES, ELEMENT_SRC)]
    srcs += [os.path.join(CSRC, h) for h in sorted(os.listdir(CSRC)) if h.endswith((".h", ".cuh"))]
    return srcs + [os.path.join(ROOT, "include", "dg.h"), os.path.abspath(__file__)]


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(LIBDIR, exist_ok=True)
    if not force and os.path.exists(LIB):
        lib_t = os.path.getmtime(LIB)
        if all(os.path.getmtime(s) <= lib_t for s in dependencies()):
            return LIB
    jobs = [(ELEMENT_SRC, f"dg_element_{n}_{p}", (f"-DDG_N={n}", f"-DDG_PART={p}")) for n, p in ELEMENT_BUILDS]
    jobs += [(s, os.path.splitext(s)[0], ()) for s in SOURCES]
    objs = [os.path.join(LIBDIR, name + ".o") for _, name, _ in jobs]
    with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
        list(ex.map(_compile, [j[0] for j in jobs], objs, [j[2] for j in jobs]))
    tmp = LIB + ".tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"linking libdg.so failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    if verbose:
        print(f"built {LIB}")
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True)
    build_probe(force="--force" in sys.argv)
