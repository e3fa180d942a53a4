"""Builds libmslt.so (the CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import re
import subprocess
import sys
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmslt.so")
SOURCES = ["mslt.cu", "gemm.cu", "gemm_simt.cu", "gemm_f32.cu", "gemm_f32x3.cu", "gemm_tc.cu", "gemm_tc_small.cu", "attn_tc.cu", "attn_f32.cu", "kernels.cu", "ops.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "mslt.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _compile(src: str, obj: str):
    return [_nvcc(), *[f for f in NVCC_FLAGS if f != "--use_fast_math=false"], "-Xptxas=-v", "-c",
            os.path.join(CSRC, src), "-o", obj]


def resource_usage(src: str) -> dict:
    """Compiles one source file and returns what ptxas reports: {mangled kernel name: (registers, spilled bytes)}."""
    with tempfile.TemporaryDirectory() as tmp:
        r = subprocess.run(_compile(src, os.path.join(tmp, "out.o")), stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if r.returncode:
        raise RuntimeError(f"nvcc failed on {src}")
    found = re.findall(r"entry function '(\w+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers",
                       r.stdout.decode(), re.S)
    return {name: (int(regs), int(stores) + int(loads)) for name, stores, loads, regs in found}


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every .cu of the library into one shared object; returns its path."""
    if not force and not needs_build():
        return LIB
    objs = []
    odir = os.path.join(HERE, "_build")
    os.makedirs(odir, exist_ok=True)
    procs = []
    for src in SOURCES:
        obj = os.path.join(odir, src.replace(".cu", ".o"))
        procs.append((src, subprocess.Popen(_compile(src, obj), stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out.decode())
        if p.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
    link = [_nvcc(), "-shared", "-o", LIB, *objs]
    r = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if r.returncode:
        sys.stderr.write(r.stdout.decode())
        raise RuntimeError("linking libmslt.so failed")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
