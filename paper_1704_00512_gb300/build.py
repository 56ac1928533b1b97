"""Build libcheb.so in-tree with nvcc for sm_103a (GB300).

Each .cu translation unit is compiled in parallel to an object under _build/,
then linked into paper_1704_00512_gb300/libcheb.so.  Rebuilds only when a
source or header is newer than the library.
"""

from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libcheb.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include")]

# Sources whose kernels fill the register file (128 registers, 512 threads a block), and
# the bytes of register spill that each kernel may have: those of the code whose times are
# stated beside it.  More would go unnoticed into the hot path, so it fails the build.
# Kernels not named here may have none.
SPILL_LIMITS = {
    "colstep.cu": {"k_colstepIfE": 12},
    "product.cu": {"k_product": 64},
}


def spills(ptxas: str) -> dict[str, int]:
    """Bytes of spill stores of every function in the output of ptxas -v."""
    out, fn = {}, None
    for line in ptxas.splitlines():
        if m := re.search(r"Function properties for (\S+)", line):
            fn = m.group(1)
        elif (m := re.search(r"(\d+) bytes spill stores", line)) and fn:
            out[fn] = int(m.group(1))
    return out


def check_spills(src: str, ptxas: str) -> None:
    """Raise if a function of src spills more than its limit."""
    limits = SPILL_LIMITS.get(os.path.basename(src))
    if limits is None:
        return
    found = spills(ptxas)
    if not found:
        raise RuntimeError(f"{src}: ptxas reported no function")
    for fn, n in found.items():
        allowed = max([b for name, b in limits.items() if name in fn], default=0)
        if n > allowed:
            raise RuntimeError(f"{src}: {fn} spills {n} bytes of registers, {allowed} allowed")


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    return "nvcc"


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps() -> list[str]:
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(d) <= t for d in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source and link libcheb.so; returns the library path."""
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src: str) -> str:
        obj = os.path.join(BUILD, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc, *ARCH, *FLAGS, "-c", src, "-o", obj]
        if os.path.basename(src) in SPILL_LIMITS:
            cmd += ["-Xptxas", "-v"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        check_spills(src, r.stderr)
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 4)) as ex:
        objs = list(ex.map(compile_one, sources()))
    tmp = LIB + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
