"""Build libst.so (the CUDA library) in-tree with nvcc for sm_103a.

The translation units are compiled in parallel and linked into
paper_2606_14480_gb300/libst.so (CUDA runtime linked statically).
"""

from __future__ import annotations

import os
import re
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libst.so")
SOURCES = ("st_seed256.cu", "st_seed256w.cu", "st_seed384.cu", "st_seed512.cu", "st_seed1024.cu", "st_seed.cu", "st_kernels.cu",
           "st_runtime.cu", "st_static.cu", "st_ut.cu")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "st.h")]
    return max(os.path.getmtime(f) for f in files)


def check_seed_registers(log: str) -> int:
    """Checks `ptxas -v` output: every k_seed<threads, registers, ..> in it
    keeps to its registers, on which the CTAs per SM and with them the launch
    shapes rest.  Returns how many it saw."""
    seen = 0
    for name, used in re.findall(r"Compiling entry function '(\S+)'.*?Used (\d+) registers", log, re.S):
        m = re.search(r"k_seedILi(\d+)ELi(\d+)E", name)
        if m:
            seen += 1
            if int(used) > int(m.group(2)):
                raise RuntimeError(f"k_seed for {m.group(1)} threads takes {used} registers a thread, "
                                   f"not {m.group(2)}: {name}")
    return seen


def build(force: bool = False, verbose: bool = False, extra=()) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    common = [nvcc(), *ARCH, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
              "-I", INCLUDE, "-I", CSRC, *extra]

    def compile_one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        seed = re.fullmatch(r"st_seed\d+w?\.cu", src)
        cmd = common + (["-Xptxas", "-v"] if seed else []) + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if seed and not check_seed_registers(r.stdout + r.stderr):
            raise RuntimeError(f"no register counts of k_seed in the compiler's output for {src}")
        return obj

    with ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "static", "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
