"""Build libpk.so in-tree with nvcc for sm_103a (GB300).

The translation units are compiled in parallel and linked against cuFFT; the
CUDA runtime is linked statically.  The result lands next to this file and is
loaded by the binding in ``__init__.py``.  Rebuilds only when a source or the
public header is newer than the library.
"""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libpk.so")
SOURCES = ["pk_kernels.cu", "pk_api.cu", "pk_static.cu", "pk_lognormal.cu", "pk_survey.cu", "pk_fft.cu", "pk_fft_zyx.cu",
           "pk_fft64.cu"]
# sources compiled several times, once per group of template instances
GROUPS = {"pk_fft_zyx.cu": ["-DPK_ZYX_GROUP=%d" % g for g in range(3)]}
HEADERS = [os.path.join(ROOT, "include", "pk.h"), os.path.join(CSRC, "pk_internal.h"),
           os.path.join(CSRC, "pk_plan.h"), os.path.join(CSRC, "pk_ylm.h"), os.path.join(CSRC, "pk_sums.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _cuda_lib_dir() -> str:
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    for sub in ("lib64", "lib", os.path.join("targets", "sbsa-linux", "lib"),
                os.path.join("targets", "x86_64-linux", "lib")):
        d = os.path.join(home, sub)
        if os.path.exists(os.path.join(d, "libcufft.so")):
            return d
    return os.path.join(home, "lib64")


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + HEADERS + [__file__]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    os.makedirs(OUT_DIR, exist_ok=True)
    nvcc = _nvcc()
    common = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off",
                     "-I", os.path.join(ROOT, "include")]
    procs = []
    objs = []
    units = [(src, g, flag) for src in SOURCES for g, flag in enumerate(GROUPS.get(src, [None]))]
    for src, g, flag in units:
        obj = os.path.join(OUT_DIR, src.replace(".cu", "%s.o" % ("" if flag is None else "_%d" % g)))
        objs.append(obj)
        cmd = [nvcc] + common + ([] if flag is None else [flag]) + ["-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    for cmd, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0:
            raise RuntimeError("nvcc failed: %s\n%s" % (" ".join(cmd), out.decode(errors="replace")))
        if verbose and out:
            print(out.decode(errors="replace"), file=sys.stderr)
    libdir = _cuda_lib_dir()
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs + [
        "-L" + libdir, "-lcufft", "-Xlinker", "-rpath," + libdir]
    if verbose:
        print(" ".join(cmd), file=sys.stderr)
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    if res.returncode != 0:
        raise RuntimeError("link failed: %s\n%s" % (" ".join(cmd), res.stdout.decode(errors="replace")))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
