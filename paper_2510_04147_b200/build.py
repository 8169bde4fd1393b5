"""Builds the C-ABI shared library from csrc/ with nvcc for sm_100a (in-tree, no JIT cache)."""
from __future__ import annotations

import os
import re
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libssd_b200.so")
SOURCES = ["elementwise.cu", "attention.cu", "attention_fill_tc.cu", "attention_verify.cu", "attention_verify_pipe.cu", "gemm.cu", "gemm_dense.cu", "gemm_wave.cu", "tree.cu", "ssd_lib.cu", "noalloc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _newer(src: str, dst: str) -> bool:
    if not os.path.exists(dst):
        return True
    t = os.path.getmtime(dst)
    deps = [src] + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".h") or f.endswith(".cuh")]
    deps.append(os.path.join(HERE, "..", "include", "ssd.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def check_register_shares(source: str, log: str) -> None:
    """Raises if a kernel of `source` that shifts registers between its warpgroups (kRegsSoftmax, kRegsOther) was compiled to fewer
    than the shares add up to: they come out of what a block is launched with, so its launcher would refuse every launch."""
    const = {k: int(v) for k, v in re.findall(r"(kThreads|kRegsSoftmax|kRegsOther) = (\d+)", source)}
    if "kRegsSoftmax" not in const:
        return
    need = 256 * const["kRegsSoftmax"] + (const["kThreads"] - 256) * const["kRegsOther"]
    used = [int(n) for n in re.findall(r"Used (\d+) registers", log)]
    if not used or min(used) * const["kThreads"] < need:
        raise RuntimeError(f"register shares of {need} need {-(-need // const['kThreads'])} registers a thread, compiled to {used}")


def build(force: bool = False, verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)

    def compile_one(name: str):
        src = os.path.join(CSRC, name)
        obj = os.path.join(OBJ, name.replace(".cu", ".o"))
        if not force and not _newer(src, obj):
            return obj, ""
        r = subprocess.run([nvcc, *NVCC_FLAGS, "-c", src, "-o", obj], capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {name}:\n{r.stdout}\n{r.stderr}")
        try:
            with open(src) as f:
                check_register_shares(f.read(), r.stderr)
        except RuntimeError:
            os.remove(obj)                         # (or the next build would take it for a good one)
            raise
        return obj, r.stderr

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    objs = [o for o, _ in results]
    if verbose:
        for _, log in results:
            if log:
                print(log, file=sys.stderr)
    if force or not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs):
        tmp = LIB + f".{os.getpid()}.tmp"         # linked beside the target, then moved: never half a library
        r = subprocess.run([nvcc, "-shared", "-o", tmp, *objs, "-gencode", "arch=compute_100a,code=sm_100a"],
                           capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
