"""Build the CUDA C-ABI library (libgkv.so) for sm_100a, in tree, with nvcc."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libgkv.so")
CALL_SOURCE = os.path.join(CSRC, "gkv_call.cpp")         # the binding's extension: a decode step's calls without ctypes
CALL_LIB = os.path.join(HERE, "_gkv_call" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["gkv_api.cu", "gkv_decode.cu", "gkv_units.cu", "gkv_pack.cu", "gkv_ingest.cu", "gkv_quest.cu", "gkv_rdplan.cu", "gkv_mla.cu", "gkv_mla_decode.cu"]
ABI = os.path.join(CSRC, "..", "..", "include", "gkv.h")
HEADERS = ["gkv_internal.h", "gkv_exchange.h", "gkv_layout.cuh", "gkv_mla.h", ABI]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def needs_build() -> bool:
    def stale(lib, deps):
        return not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in deps)
    own = os.path.abspath(__file__)
    return stale(LIB, [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [own]) or stale(CALL_LIB, [CALL_SOURCE, ABI, own])


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    objs = []
    flags = list(NVCC_FLAGS)
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    # (the extension first: it is compiled against the ABI, and an interrupted build must not leave an old one beside a new library)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-I{sysconfig.get_path('include')}",
                    CALL_SOURCE, "-o", CALL_LIB], check=True)
    cmd = [_nvcc(), "-shared", "-o", LIB, *objs, "-Xcompiler", "-fPIC", "-lpthread"]
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
