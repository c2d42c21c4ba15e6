"""Compile libipd.so in-tree for sm_103a (nvcc; one translation unit per .cu,
compiled in parallel, linked into a shared library with the CUDA runtime
linked statically), and the Python binding's extension module beside it."""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT_DIR = os.path.join(HERE, "_lib")
LIB = os.path.join(OUT_DIR, "libipd.so")
NATIVE = os.path.join(OUT_DIR, "_ipd_native.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall",
         "--expt-relaxed-constexpr"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _defines():
    """Build-time switches from the environment.  IPD_TC_MIN_ROWS (default 4)
    moves the row count from which attention tasks use the tensor cores; it
    exists to measure the crossover between the two paths."""
    v = os.environ.get("IPD_TC_MIN_ROWS")
    return [f"-DIPD_TC_MIN_ROWS={int(v)}"] if v else []


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(OUT_DIR, exist_ok=True)
    srcs = sources()
    native_src = os.path.join(CSRC, "native.cpp")
    deps = srcs + [native_src] + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")] + \
        [os.path.join(HERE, "..", "include", "ipd.h")]
    defines = _defines()
    stamp = os.path.join(OUT_DIR, "defines.txt")
    same_defines = os.path.exists(stamp) and open(stamp).read() == " ".join(defines)
    if not force and same_defines and os.path.exists(LIB) and os.path.exists(NATIVE):
        t = os.path.getmtime(NATIVE)  # written last
        if all(os.path.getmtime(d) <= t for d in deps):
            return LIB
    nvcc = _nvcc()
    objs = []

    def compile_one(src):
        obj = os.path.join(OUT_DIR, os.path.basename(src)[:-3] + ".o")
        cmd = [nvcc, *ARCH, *FLAGS, *defines, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        objs = list(ex.map(compile_one, srcs))
    tmp = LIB + ".tmp"
    r = subprocess.run([nvcc, *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    # the extension links against the library in its own folder
    tmp = NATIVE + ".tmp"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-fPIC", "-shared", "-fvisibility=hidden",
                        "-I", sysconfig.get_paths()["include"], native_src, "-o", tmp,
                        "-L", OUT_DIR, "-l:libipd.so", "-Wl,-rpath,$ORIGIN"],
                       capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"the binding's extension failed to build:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, NATIVE)
    with open(stamp, "w") as f:
        f.write(" ".join(defines))
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
