"""Builds libss.so (the C-ABI library) in-tree for sm_103a with nvcc.

The translation units (FP32 kernels, FP64 kernels, host runtime, one unit per length and type of the
two-pass transforms) compile in parallel and link into ``paper_1804_07135_gb300/libss.so`` against the shared CUDA runtime.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libss.so")
SOURCES = ("ss_kernels_f32.cu", "ss_kernels_f64.cu", "ss_api.cu", "ss_noalloc.cu")
# lengths of the two-pass transforms (SS_T2_LENGTHS of csrc/ss_internal.h)
T2_LENGTHS = (32, 48, 64, 80, 96, 112, 128, 144, 160, 192, 224, 256, 288, 320, 384, 448, 512)
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    cand = [os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc"), shutil.which("nvcc") or ""]
    for c in cand:
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found (set CUDA_HOME)")


def cuda_lib_dir() -> str:
    home = os.path.dirname(os.path.dirname(nvcc()))
    for d in ("lib64", "lib", os.path.join("targets", "sbsa-linux", "lib"), os.path.join("targets", "x86_64-linux", "lib")):
        p = os.path.join(home, d)
        if os.path.exists(os.path.join(p, "libcudart.so")):
            return p
    return os.path.join(home, "lib64")


def _deps() -> list[str]:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "ss.h"))
    files.append(os.path.abspath(__file__))
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _deps())


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    common = [cc, *ARCH, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]

    def compile_one(unit) -> str:
        src, defines = unit
        obj = os.path.join(BUILD, "_".join([src[:-3], *(str(v) for v in defines.values())]) + ".o")
        cmd = common + [f"-D{k}={v}" for k, v in defines.items()] + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    units = [(src, {}) for src in SOURCES]
    units += [("ss_twopass.cu", {"SS_T2_P": P, "SS_T2_T": T}) for P in reversed(T2_LENGTHS) for T in ("double", "float")]
    with cf.ThreadPoolExecutor(min(len(units), os.cpu_count() or 8)) as ex:
        objs = list(ex.map(compile_one, units))
    tmp = LIB + f".tmp{os.getpid()}"
    libdir = cuda_lib_dir()
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *objs, "-cudart", "shared", "-L", libdir,
           "-Xlinker", "-rpath", "-Xlinker", libdir]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
