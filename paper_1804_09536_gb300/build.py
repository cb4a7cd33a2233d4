"""Build the in-tree shared library ``libtfft.so`` (C ABI of include/tfft.h).

Compiles the CUDA kernels and the host plan code for sm_103a with nvcc, one
process per translation unit in parallel, and links them into
``paper_1804_09536_gb300/libtfft.so``.  No cmake, no setuptools.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libtfft.so")

SOURCES = ["tfft_kernels.cu", "tfft_spec.cu", "tfft_spec_real.cu", "tfft_tma.cu", "tfft_noalloc.cu", "tfft_pointwise.cu", "tfft_batch.cu", "tfft_tc.cu", "tfft_tc_strided.cu", "tfft_blue.cu", "tfft_plan.cpp", "tfft_exchange.cpp",
           "tfft_tmageo.cpp", "tfft_exec.cpp", "tfft_hostio.cpp", "tfft_batch_host.cpp"]
# the specialised passes, one object per part of their table (kSpecParts in tfft_spec_pass.cuh; no row is in part 0)
PARTS = {"tfft_spec_part.cu": [("TFFT_SPEC_PART", k) for k in range(1, 11)]}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _units():
    """(source file, object name, extra flags) of every translation unit."""
    for src in SOURCES:
        yield src, src + ".o", []
    for src, parts in PARTS.items():
        for name, k in parts:
            yield src, f"{src}.{k}.o", [f"-D{name}={k}"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _flags(ptxas_verbose: bool):
    f = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-O3", "-I", INCLUDE, "-I", CSRC,
         "--expt-relaxed-constexpr"] + ARCH
    if ptxas_verbose:
        f += ["-Xptxas", "-v"]
    return f


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False, ptxas_verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    headers = [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith((".h", ".cuh", ".map"))]
    headers.append(os.path.join(INCLUDE, "tfft.h"))
    procs, objs = [], []
    for src, oname, extra in _units():
        path = os.path.join(CSRC, src)
        obj = os.path.join(BUILD, oname)
        objs.append(obj)
        if force or _stale(obj, [path] + headers):
            cmd = [nvcc(), "-c", path, "-o", obj] + _flags(ptxas_verbose) + extra
            if src.endswith(".cpp"):
                cmd[1:1] = ["-x", "c++"]
            if verbose:
                print(" ".join(cmd), flush=True)
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = []
    for src, pr in procs:
        out, _ = pr.communicate()
        text = out.decode(errors="replace")
        if pr.returncode != 0:
            failed.append((src, text))
        elif verbose and text.strip():
            print(text, flush=True)
    if failed:
        msg = "\n".join(f"--- {s} ---\n{t}" for s, t in failed)
        raise RuntimeError(f"nvcc failed:\n{msg}")
    if force or _stale(LIB, objs):
        cmd = [nvcc(), "-shared", "-o", LIB + ".tmp"] + objs + ARCH + [
            "-cudart", "static", "-Xlinker", "--version-script=" + os.path.join(CSRC, "exports.map")]
        if verbose:
            print(" ".join(cmd), flush=True)
        r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n" + r.stdout.decode(errors="replace"))
        os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    build(verbose=True, force="--force" in sys.argv, ptxas_verbose="-v" in sys.argv)
