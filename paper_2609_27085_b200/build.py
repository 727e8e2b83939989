"""Builds libcrossflow_attn.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _marshal.<abi>.so (the CPython
extension that marshals the arguments of the hot entry points) with g++ and the running interpreter's headers.

    python -m paper_2609_27085_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The library links the static CUDA runtime, so it can be
loaded (and its symbols listed) on a machine with no driver; any CUDA call there fails with a
status code instead.  Extra nvcc flags (a -D for a development build) are taken from CF_NVCC_EXTRA.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcrossflow_attn.so")
# CPython extension: argument marshalling of the hot entry points.  The name carries the interpreter's ABI tag, so that another
# interpreter misses the file instead of loading it; building it takes that interpreter's headers.
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["api.cu", "plan.cpp", "kv_append.cu", "decode_splitk.cu", "prefill_tc.cu", "prefill_tc2.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale() -> bool:
    if not (os.path.exists(LIB) and os.path.exists(MARSHAL)):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(MARSHAL))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [
        os.path.join(HERE, "..", "include", "crossflow_attn.h"), os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    # both results are built under temporary names, put in place together and never left behind
    tmp_marshal, tmp = MARSHAL + f".tmp{os.getpid()}", LIB + f".tmp{os.getpid()}"
    try:
        procs, objs = [], []
        for src in SOURCES:
            obj = os.path.join(objdir, os.path.splitext(src)[0] + ".o")
            objs.append(obj)
            cmd = [_nvcc(), *NVCC_FLAGS, *os.environ.get("CF_NVCC_EXTRA", "").split(), "-c", os.path.join(CSRC, src), "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wall", "-I", sysconfig.get_paths()["include"],
               os.path.join(CSRC, "marshal.cpp"), "-o", tmp_marshal]
        procs.append(("marshal.cpp", subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        failed = []
        for src, p in procs:
            out, _ = p.communicate()
            if p.returncode != 0 or verbose:
                sys.stderr.write(f"--- {src}\n{out}\n")
            if p.returncode != 0:
                failed.append(src)
        if failed:
            raise RuntimeError(f"compilation failed: {', '.join(failed)}")
        subprocess.check_call([_nvcc(), "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", tmp, *objs,
                               "-cudart", "static"])
        os.replace(tmp, LIB)
        os.replace(tmp_marshal, MARSHAL)
    finally:
        for path in (tmp, tmp_marshal):
            if os.path.exists(path):
                os.remove(path)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
