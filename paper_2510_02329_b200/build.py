"""Compile the CUDA library in-tree for sm_100a (no JIT cache: the .so sits beside this file)."""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "sj_api.cu")
INST = os.path.join(HERE, "csrc", "sj_mega_inst.cu")
LIB = os.path.join(HERE, "libsjverify.so")


def units():
    """(name, source, macros) of every object file: the library, and the persistent kernel's instantiations
    (minutes of compile time in one translation unit) by head dimension and timeline code."""
    out = [("sj_api", SRC, [])]
    for hd in (64, 128):
        for trace in (0, 1):
            name = f"mega_kernel_{hd}" + ("_trace" if trace else "")
            out.append((name, INST, [f"-DSJ_INST_NAME={name}", f"-DSJ_INST_HD={hd}", f"-DSJ_INST_TRACE={trace}"]))
    return out


def deps():
    """Every file the library is compiled from: all of csrc/ plus the public header."""
    src = sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")) + glob.glob(os.path.join(HERE, "csrc", "*.cuh")))
    return src + [os.path.join(os.path.dirname(HERE), "include", "sj.h")]


def lib_path() -> str:
    return LIB


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in deps())


def _nvcc(args, verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", *args], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + r.stdout + r.stderr)
    if verbose:
        print(r.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    flags = ["-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"] + (["-Xptxas", "-v"] if verbose else [])
    with tempfile.TemporaryDirectory() as tmp:
        objs = {name: os.path.join(tmp, name + ".o") for name, _, _ in units()}
        with concurrent.futures.ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as pool:
            jobs = [pool.submit(_nvcc, [*flags, *macros, "-c", "-o", objs[name], src], verbose)
                    for name, src, macros in units()]
            for j in jobs:
                j.result()
        _nvcc(["-shared", "-o", LIB, *objs.values()], False)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
