"""Build libgrid_dwf.so in-tree with nvcc for sm_103a (GB300).

Each translation unit under csrc/ is compiled in its own nvcc process (``dhop_packed.cu`` once per
storage precision and number of slice pairs), in parallel, then linked into
``paper_2203_06777_gb300/lib/libgrid_dwf.so`` with a shared CUDA runtime. A rebuild happens only when a
source or header is newer than the library.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import re
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIBDIR = os.path.join(PKG, "lib")
LIB = os.path.join(LIBDIR, "libgrid_dwf.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
                     "--expt-relaxed-constexpr"]


def nvcc_path() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build libgrid_dwf.so")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _units():
    """(source, object name, extra flags) of every translation unit, the slowest first."""
    with open(os.path.join(CSRC, "dhop_kernel.cuh")) as f:
        pairs = re.search(r"#define DWF_PAIR_SPECIALISATIONS\(M\)(.*)", f.read()).group(1)
    units = []
    for src in _sources():
        name = os.path.basename(src)[:-3]
        if name != "dhop_packed":
            units.append((src, name, []))
            continue
        for n in ["0"] + re.findall(r"M\((\d+)\)", pairs):
            for prec in ("P32", "P16", "PB16"):
                units.insert(0, (src, f"{name}_{prec}_{n}", [f"-DDWF_PREC={prec}", f"-DDWF_PAIRS={n}"]))
    return units


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(ROOT, "include", "grid_dwf.h"),
                                                                   os.path.abspath(__file__)]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(d) <= t for d in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile (if needed) and return the path of libgrid_dwf.so."""
    if not force and up_to_date():
        return LIB
    nvcc = nvcc_path()
    os.makedirs(BUILD, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)

    def compile_unit(unit):
        src, name, flags = unit
        obj = os.path.join(BUILD, name + ".o")
        cmd = [nvcc] + NVCC_FLAGS + flags + ["-c", src, "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
        out = r.stdout.decode(errors="replace")
        if verbose and out:
            print(out, file=sys.stderr)
        return obj, f"{name}:\n{out}" if r.returncode != 0 else None

    with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 4) as pool:
        done = list(pool.map(compile_unit, _units()))
    objs = [obj for obj, _ in done]
    errors = [e for _, e in done if e]
    if errors:
        raise RuntimeError("nvcc failed:\n" + "\n".join(errors))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc] + ARCH + ["-shared", "-cudart", "shared", "-o", tmp] + objs
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
