"""Builds libpurekv.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _marshal, the Python module that passes
arguments to it (its file name carries the interpreter's ABI, so another Python builds its own).

    python -m paper_2510_25600_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB = os.path.join(_HERE, "libpurekv.so")
MARSHAL = os.path.join(_HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["plan.cu", "compact.cu", "decode.cu", "select.cu", "score.cu", "score_tc.cu", "prefill.cu", "prefill_simt.cu", "prefill_tc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(INCLUDE, "purekv.h"))
    objdir = os.path.join(_HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
    if verbose:
        flags += ["-Xptxas", "-v"]
    objs, procs = [], []
    for src in SOURCES:
        sp = os.path.join(CSRC, src)
        ob = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(ob)
        if force or _stale(ob, [sp] + headers):
            cmd = [_nvcc(), *flags, "-I", INCLUDE, "-I", CSRC, "-c", sp, "-o", ob]
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if force or procs or _stale(LIB, objs):
        subprocess.check_call([_nvcc(), "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"])
    src = os.path.join(CSRC, "marshal.cpp")
    untagged = os.path.join(_HERE, "_marshal.so")  # of an earlier build: any interpreter would load it
    if os.path.exists(untagged) and untagged != MARSHAL:
        os.remove(untagged)
    if force or _stale(MARSHAL, [src, LIB] + headers):
        # found beside the module at run time: one copy of the library, whether it is loaded through this or by path
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-I", INCLUDE,
                               src, "-o", MARSHAL, "-L", _HERE, "-l:libpurekv.so", "-Wl,-rpath,$ORIGIN"])
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
