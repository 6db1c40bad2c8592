"""Build the CUDA library libdsrg.so in-tree for sm_103a with nvcc."""
from __future__ import annotations

import os
import re
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libdsrg.so")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
         "--expt-relaxed-constexpr", "-I" + os.path.join(os.path.dirname(HERE), "include")]


def nvcc() -> str:
    for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def check_registers(source: str, log: str) -> None:
    """The split kernel's warpgroups move registers between them (setmaxnreg)
    within the total that the block is launched with, so every instantiation
    has to be compiled to exactly the count that the source states."""
    want = int(re.search(r"constexpr int OZ_REGS = (\d+)", source).group(1))
    used = re.findall(r"Compiling entry function '(\S*k_ozaki_mma\S*)'.*?Used (\d+) registers", log, re.S)
    if not used:
        raise RuntimeError("ptxas reported no registers for k_ozaki_mma")
    bad = [f"{name}: {n}" for name, n in used if int(n) != want]
    if bad:
        raise RuntimeError(f"k_ozaki_mma needs {want} registers a thread, compiled to " + ", ".join(bad))


def _newer(target, deps):
    if not os.path.exists(target):
        return False
    t = os.path.getmtime(target)
    return all(os.path.getmtime(d) <= t for d in deps)


def build(force: bool = False, verbose: bool = False, extra_flags=None) -> str:
    os.makedirs(BUILD, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(os.path.dirname(HERE), "include", "dsrg.h"))
    cc = nvcc()
    flags = FLAGS + list(extra_flags or [])

    def compile_one(src):
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        if not force and _newer(o, [s] + headers):
            return o
        ptxas = ["-Xptxas", "-v"] if src == "ozaki.cu" else []
        cmd = [cc] + ARCH + flags + ptxas + ["-c", s, "-o", o]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if ptxas:
            try:
                with open(s) as f:
                    check_registers(f.read(), r.stdout + r.stderr)
            except RuntimeError:
                os.remove(o)
                raise
        if verbose and r.stderr:
            print(r.stderr, file=sys.stderr)
        return o

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    if force or not _newer(LIB, objs):
        cmd = [cc] + ARCH + ["-shared", "--cudart", "static", "-o", LIB] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
