"""Build step: compile the CUDA library for sm_100a into the package directory."""
from __future__ import annotations

import fcntl
import hashlib
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfh_sm100a.so")
SOURCES = [os.path.join(CSRC, f) for f in ("fh_warp_f32.cu", "fh_warp_bf16.cu", "fh_warp_f32_plain.cu", "fh_warp_bf16_plain.cu",
                                          "fh_warp_f32_random.cu", "fh_warp_bf16_random.cu", "fh_cta_f32.cu", "fh_cta_bf16.cu",
                                          "fh_generic.cu", "fh_decompress.cu", "fh.cu", "fh_plan.cpp")]
HEADERS = [os.path.join(CSRC, f) for f in ("fh_device.cuh", "fh_blocks.cuh", "fh_channel.cuh", "fh_compress.cuh",
                                          "fh_decompress.cuh", "fh_launch.cuh", "fh_launch_cta.cuh",
                                          "fh_launch_warp.cuh")] + \
    [os.path.join(os.path.dirname(HERE), "include", "fh.h")]
DEPS = SOURCES + HEADERS + [os.path.abspath(__file__)]    # (this file: the flags)
OBJDIR = os.path.join(HERE, "_build")
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC",
         "--fmad=false"]


def _run(cmd, out: str, what: str) -> str:
    """Runs a compiler that writes `out`, which appears only when it is complete; returns what it said."""
    part = f"{out}.{os.getpid()}.tmp"
    r = subprocess.run(["nvcc", *FLAGS, *cmd, "-o", part], capture_output=True, text=True)
    if r.returncode != 0:
        if os.path.exists(part):
            os.remove(part)
        raise RuntimeError(f"{what} failed:\n" + r.stderr)
    os.replace(part, out)
    return r.stderr


def _object_path(source: str) -> str:
    """Objects carry the flags they were made with in their names."""
    return os.path.join(OBJDIR, f"{os.path.basename(source)}.{hashlib.sha256(' '.join(FLAGS).encode()).hexdigest()[:12]}.o")


def _object(source: str, extra) -> str:
    """Compiles one source when its object is missing or older; returns what the compiler said."""
    obj = _object_path(source)
    t = os.path.getmtime(obj) if os.path.exists(obj) else -1.0
    if not extra and all(os.path.getmtime(f) <= t for f in [source] + HEADERS):
        return ""
    return _run([*extra, "-c", source], obj, "nvcc")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile when the library is missing or older than a source or this file; the sources compile side by side, one
    build at a time.  Returns the library path."""
    if not force and os.path.exists(LIB):
        t = os.path.getmtime(LIB)
        if all(os.path.getmtime(d) <= t for d in DEPS):
            return LIB
    os.makedirs(OBJDIR, exist_ok=True)
    with open(os.path.join(OBJDIR, "lock"), "w") as lock:
        fcntl.flock(lock, fcntl.LOCK_EX)
        if force:
            for f in os.listdir(OBJDIR):
                if f != "lock":
                    os.remove(os.path.join(OBJDIR, f))
        extra = ["-Xptxas", "-v"] if verbose else []
        with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as pool:
            said = list(pool.map(lambda s: _object(s, extra), SOURCES))
        if verbose:
            sys.stderr.write("".join(said))
        _run(["-shared", *map(_object_path, SOURCES)], LIB, "linking")
    return LIB


if __name__ == "__main__":    # from the command line: everything anew
    print(build(force=True, verbose="-v" in sys.argv))
