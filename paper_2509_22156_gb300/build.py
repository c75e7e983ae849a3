"""Builds libpit.so in-tree with nvcc for sm_103a (GB300).

Translation units are compiled in parallel, then linked into a shared
library next to this file.  No CMake; runs on the CPU-only build machine
(cross-compilation) and on the GPU machine (Arm host) alike.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libpit.so")
SOURCES = ["pit_phi_heat_pair.cu", "pit_phi_varheat_pair.cu"] + \
    [f"pit_direct_{p}.cu" for p in ("mixed", "pair")] + ["pit_fixed.cu"] + \
    [f"pit_phi_{op}_{p}.cu" for op in ("heat", "varheat", "ou", "lsde", "cme") for p in ("mixed", "fp64", "fp32")] + \
    [f"pit_net_d{d}.cu" for d in range(1, 7)] + ["pit_phi.cu", "pit_cluster.cu", "pit_net.cu", "pit_aux.cu", "pit_recomb.cu", "pit_api.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libpit.so")


def _stale(obj: str, deps: list[str]) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra: list[str] | None = None) -> str:
    os.makedirs(BUILD, exist_ok=True)
    nv = nvcc()
    headers = [os.path.join(CSRC, "pit_internal.cuh"), os.path.join(CSRC, "pit_phi.cuh"),
               os.path.join(CSRC, "pit_direct.cuh"), os.path.join(CSRC, "pit_fixed.cuh"),
               os.path.join(CSRC, "pit_net.cuh"), os.path.join(ROOT, "include", "pit.h")]
    flags = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
                    "-I", os.path.join(ROOT, "include")] + (extra or [])
    procs, objs = [], []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(BUILD, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [nv] + flags + ["-c", s, "-o", o]
            if verbose:
                print(" ".join(cmd), file=sys.stderr)
            procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = []
    for cmd, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0:
            failed.append((cmd, out.decode(errors="replace")))
        elif verbose and out:
            print(out.decode(errors="replace"), file=sys.stderr)
    if failed:
        msg = "\n".join(" ".join(c) + "\n" + o for c, o in failed)
        raise RuntimeError("nvcc failed:\n" + msg)
    if force or procs or _stale(LIB, objs):
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nv] + ARCH + ["-shared", "-o", tmp] + objs + ["-lcudart"]
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
