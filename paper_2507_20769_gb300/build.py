"""Build libivb.so in-tree with nvcc for sm_103a (GB300).

Usage: python -m paper_2507_20769_gb300.build [--force]
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libivb.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

SOURCES = ["ivb_kernels.cu", "ivb_api.cu", "ivb_probe.cu", "ivb_static.cu", "ivb_compile.cpp", "ivb_bnb.cpp",
           "ivb_jit.cpp", "ivb_jit_seg.cpp", "ivb_host.cpp"]
HEADERS = ["ivb_internal.h", "ivb_iv.cuh", "ivb_fixed.cuh", "ivb_fp64x.cuh", "ivb_emu.cuh", "ivb_kparams.h",
           "ivb_bound_common.cuh", "ivb_kernels.h",
           "ivb_problem.h", "ivb_launch.h", "ivb_jit.h", "ivb_host.h", "ivb_compile.h"]
# device headers the tape-specialised kernels are compiled against at run time (NVRTC)
JIT_HEADERS = ["ivb_bound_common.cuh", "ivb_internal.h", "ivb_iv.cuh", "ivb_fixed.cuh", "ivb_fp64x.cuh", "ivb_emu.cuh",
               "ivb_kparams.h"]

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "--fmad=false", "-Xcompiler", "-fPIC",
              "-Xcompiler", "-ffp-contract=off", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libivb.so")


def _cuda_lib_dir(nvcc: str) -> str:
    home = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    for sub in ("lib64", "lib"):
        d = os.path.join(home, sub)
        if os.path.exists(os.path.join(d, "libnvrtc.so")):
            return d
    raise RuntimeError(f"libnvrtc.so not found under {home}")


def _write_jit_headers() -> None:
    """C++ arrays with the device headers' text, for NVRTC at run time."""
    names, texts = [], []
    for h in JIT_HEADERS:
        with open(os.path.join(CSRC, h)) as fh:
            text = fh.read()
        if ')IVBJIT"' in text:
            raise RuntimeError(f"{h} contains the raw-string delimiter")
        names.append(f'"{h}"')
        texts.append('R"IVBJIT(' + text + ')IVBJIT"')
    out = ("// generated by build.py from csrc/: device headers of the tape-specialised kernels\n"
           "static const char* const kJitHeaderNames[] = {" + ", ".join(names) + "};\n"
           "static const char* const kJitHeaderSources[] = {\n" + ",\n".join(texts) + "};\n")
    path = os.path.join(BUILD, "ivb_jit_headers.inc")
    old = open(path).read() if os.path.exists(path) else None
    if old != out:
        with open(path, "w") as fh:
            fh.write(out)


def _newest_input() -> float:
    paths = [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [os.path.join(INCLUDE, "ivb.h"), __file__]
    return max(os.path.getmtime(p) for p in paths if os.path.exists(p))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_input():
        return LIB
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)
    _write_jit_headers()
    cuda_lib = _cuda_lib_dir(nvcc)

    def compile_one(src):
        obj = os.path.join(BUILD, src + ".o")
        cmd = [nvcc] + ARCH + NVCC_FLAGS + ["-c", os.path.join(CSRC, src), "-o", obj]
        if src.endswith(".cpp"):
            cmd = [nvcc] + NVCC_FLAGS + ["-I", BUILD, "-x", "c++", "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stdout.write(r.stderr)
        return obj

    srcs = [s for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]
    with cf.ThreadPoolExecutor(max_workers=len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    tmp = LIB + ".tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs + ["-L", cuda_lib, "-lnvrtc", "-lnvJitLink", "-Xlinker",
                                                           "-rpath=" + cuda_lib,
                                                           "-lcudart_static", "-lrt", "-lpthread", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
