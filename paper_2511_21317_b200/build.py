"""Build libhttm.so (CUDA, sm_100a) in-tree with nvcc.

    python -m paper_2511_21317_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The library links the static CUDA runtime, so it
has no dependency on torch's copy.
"""
from __future__ import annotations

import os
import re
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libhttm.so")
OBJ_DIR = os.path.join(HERE, "_build")
SOURCES = ["httm_api.cu", "httm_small_blocks.cu", "httm_mid_blocks.cu", "httm_mem_kernels.cu", "httm_attention_tc.cu", "httm_big_blocks.cu", "httm_linear.cu", "httm_static.cu",
           "httm_umma_selftest.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
]

# Their kernels change the registers of their warps as they run (setmaxnreg).  A function that is called does not know how many its caller has
# left: in such a file everything has to be inlined.
NO_CALLS = ("httm_big_blocks.cu",)


def called_functions(ptxas_log: str) -> list[str]:
    """The device functions, other than kernels, for which ptxas -v lists properties: those that were not inlined everywhere."""
    kernels = set(re.findall(r"Compiling entry function '([^']+)'", ptxas_log))
    return [name for name in re.findall(r"Function properties for (\S+)", ptxas_log) if name not in kernels]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _deps_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "httm.h"), __file__]
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps_mtime():
        return LIB
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()
    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-Xptxas", "-v", "-I", INCLUDE, "-c", os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        if src in NO_CALLS and called_functions(res.stdout + res.stderr):
            raise RuntimeError(f"{src}: not inlined: {called_functions(res.stdout + res.stderr)}")
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".{os.getpid()}.tmp"
    subprocess.check_call([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
