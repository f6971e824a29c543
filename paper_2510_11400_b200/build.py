"""Build step: compile the CUDA library for sm_100a into the package directory."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfh_sm100a.so")
SOURCES = [os.path.join(CSRC, f) for f in ("fh.cu", "fh_warp_f32.cu", "fh_warp_bf16.cu", "fh_cta_f32.cu", "fh_cta_bf16.cu",
                                          "fh_generic.cu", "fh_decompress.cu", "fh_plan.cpp")]
HEADERS = [os.path.join(CSRC, f) for f in ("fh_device.cuh", "fh_blocks.cuh", "fh_channel.cuh", "fh_compress.cuh",
                                          "fh_decompress.cuh", "fh_launch.cuh", "fh_launch_cta.cuh",
                                          "fh_launch_warp.cuh")] + \
    [os.path.join(os.path.dirname(HERE), "include", "fh.h")]
DEPS = SOURCES + HEADERS
OBJDIR = os.path.join(HERE, "_build")
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC",
         "--fmad=false"]


def _object(source: str, extra) -> str:
    """Compiles one source when its object is missing or older; returns what the compiler said."""
    obj = os.path.join(OBJDIR, os.path.basename(source) + ".o")
    t = os.path.getmtime(obj) if os.path.exists(obj) else -1.0
    if not extra and all(os.path.getmtime(f) <= t for f in [source] + HEADERS):
        return ""
    r = subprocess.run(["nvcc", *FLAGS, *extra, "-c", source, "-o", obj], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + r.stderr)
    return r.stderr


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile when the library is missing or older than a source; the sources compile side by side.
    Returns the library path."""
    if not force and os.path.exists(LIB):
        t = os.path.getmtime(LIB)
        if all(os.path.getmtime(d) <= t for d in DEPS):
            return LIB
    os.makedirs(OBJDIR, exist_ok=True)
    if force:
        for f in os.listdir(OBJDIR):
            os.remove(os.path.join(OBJDIR, f))
    extra = ["-Xptxas", "-v"] if verbose else []
    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
        said = list(pool.map(lambda s: _object(s, extra), SOURCES))
    if verbose:
        sys.stderr.write("".join(said))
    objs = [os.path.join(OBJDIR, os.path.basename(s) + ".o") for s in SOURCES]
    r = subprocess.run(["nvcc", *FLAGS, "-shared", "-o", LIB, *objs], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("linking failed:\n" + r.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="-f" in sys.argv, verbose="-v" in sys.argv))
