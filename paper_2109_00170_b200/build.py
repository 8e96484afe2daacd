"""Build libalcs.so (the C-ABI library with the sm_100a kernels) in-tree with nvcc, and _alcs_call, a helper of the
Python binding, with gcc (the binding works without it: its calls then take 2 us longer).

    python -m paper_2109_00170_b200.build [--force]

nvcc cross-compiles for sm_100a without a GPU.  The shared object is written next to this
file; object files go to paper_2109_00170_b200/_build/.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libalcs.so")
# The binding's most frequent calls, marshalled in C; the name carries the Python it is for, so that no other one loads it.
CALL = os.path.join(PKG, "_alcs_call" + sysconfig.get_config_var("EXT_SUFFIX"))

SOURCES = ["alcs_pack.cpp", "alcs_device.cu", "alcs_conv2d.cu", "alcs_project.cu", "alcs_gather.cu", "alcs_probe.cu", "alcs_tc.cu", "alcs_tc16.cu", "alcs_tc_prep.cu", "alcs_variants_f32_g4.cu",
           "alcs_variants_f32_other.cu", "alcs_variants_f16.cu", "alcs_variants_f16_mma.cu", "alcs_variants_bf16.cu"]
HEADERS = ["alcs_internal.h", "alcs_kernels.cuh", "alcs_mma.cuh", "alcs_conv2d.cuh", "alcs_gather.h", "alcs_tc.h", "alcs_tc.cuh", "alcs_tc_prep.h"]

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC,-Wall,-fvisibility=hidden", "-I", os.path.join(ROOT, "include"),
              "-I", CSRC]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found")


def _newest_dep() -> float:
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    deps += [os.path.join(ROOT, "include", "alcs.h"), os.path.abspath(__file__)]
    return max(os.path.getmtime(d) for d in deps)


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(OBJ, os.path.splitext(src)[0] + ".o")
    srcp = os.path.join(CSRC, src)
    hdr_time = max(os.path.getmtime(os.path.join(CSRC, h)) for h in HEADERS)
    hdr_time = max(hdr_time, os.path.getmtime(os.path.join(ROOT, "include", "alcs.h")),
                   os.path.getmtime(os.path.abspath(__file__)))
    if os.path.exists(obj) and os.path.getmtime(obj) >= max(os.path.getmtime(srcp), hdr_time):
        return obj
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-x", "cu", "-c", srcp, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
    return obj


def _build_call(force: bool) -> None:
    """Compile _alcs_call if stale.  Without a C compiler or Python's headers there is none, which costs time alone."""
    src = os.path.join(CSRC, "alcs_call.c")
    if not force and os.path.exists(CALL) and os.path.getmtime(CALL) >= os.path.getmtime(src):
        return
    if os.path.exists(CALL):        # (a stale one is not left behind, whatever happens)
        os.remove(CALL)
    tmp = CALL + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-Wall", "-I", sysconfig.get_paths()["include"], src, "-o", tmp]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
        failed = f"{r.stdout}\n{r.stderr}" if r.returncode != 0 else None
    except OSError as e:
        failed = str(e)
    if failed is not None:
        print(f"_alcs_call not built, calls will go through ctypes: {failed}", file=sys.stderr)
        return
    os.replace(tmp, CALL)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile (if stale) and return the path of libalcs.so."""
    lib = _build_lib(force, verbose)
    _build_call(force)
    return lib


def _build_lib(force: bool, verbose: bool) -> str:
    os.makedirs(OBJ, exist_ok=True)
    if force:
        for f in os.listdir(OBJ):
            if f.endswith(".o"):
                os.remove(os.path.join(OBJ, f))
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_dep():
        return LIB
    with cf.ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 2)) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose), SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a",
                                                     "-cudart", "static", "-Xcompiler", "-fPIC", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
