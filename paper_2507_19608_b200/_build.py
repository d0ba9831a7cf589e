"""Builds libdelta_attn.so (sm_100a) in-tree with nvcc.  No JIT cache, no torch extension:
the library has a plain C ABI and is loaded with ctypes."""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdelta_attn.so")
LIB_DEBUG = os.path.join(HERE, "libdelta_attn_dbg.so")      # the same sources with -DDELTA_DEBUG_BOUNDS
# CPython entry points over the library: compiled against this interpreter's headers, so its file carries the
# interpreter's ABI tag and another version of Python builds its own
CALLS = os.path.join(HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
CALLS_SOURCE = "py_calls.cpp"
SOURCES = ["api.cu", "k1_delta_construct.cu", "k2_hybrid_attn_f32.cu", "k2_hybrid_attn_tc.cu", "k2_hybrid_attn_tcq.cu",
           "k3_decode_step.cu", "k3_decode_step_mma.cu", "k3_decode_step_f32.cu", "k3_decode_step_key.cu", "k1_pack_keys.cu", "decode_noalloc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "-DDELTA_BUILDING_LIB"]
LINK_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "--shared", "-lcuda"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the delta-attention library cannot be built")


def _stale(lib: str) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != CALLS_SOURCE]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "delta_attn.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps)


def build_calls(force: bool = False) -> str:
    """Compile the CPython entry points (g++, no CUDA) if missing or older than their source."""
    src = os.path.join(CSRC, CALLS_SOURCE)
    if not force and os.path.exists(CALLS) and os.path.getmtime(CALLS) >= os.path.getmtime(src):
        return CALLS
    cmd = [os.environ.get("CXX") or shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC",
           "-fvisibility=hidden", "-I", sysconfig.get_paths()["include"], "-o", CALLS + ".tmp", src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("g++ failed:\n" + r.stdout + r.stderr)
    os.replace(CALLS + ".tmp", CALLS)
    return CALLS


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """Compile the library if it is missing or older than its sources; returns its path.
    debug_bounds: the bounds-checking build (libdelta_attn_dbg.so, -DDELTA_DEBUG_BOUNDS)."""
    lib = LIB_DEBUG if debug_bounds else LIB
    if not force and not _stale(lib):
        return lib
    flags = NVCC_FLAGS + (["-DDELTA_DEBUG_BOUNDS"] if debug_bounds else []) + (["-Xptxas", "-v"] if verbose else [])
    nvcc = _nvcc()

    def run(cmd: list) -> str:
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + r.stdout + r.stderr)
        return r.stderr

    # the files side by side: they share no device symbols, and one nvcc call would compile them in turn
    with tempfile.TemporaryDirectory() as tmp, ThreadPoolExecutor(os.cpu_count()) as pool:
        objs = [os.path.join(tmp, s + ".o") for s in SOURCES]
        logs = list(pool.map(run, [[nvcc, *flags, "-c", os.path.join(CSRC, s), "-o", o] for s, o in zip(SOURCES, objs)]))
        run([nvcc, *LINK_FLAGS, "-o", lib + ".tmp", *objs])
    os.replace(lib + ".tmp", lib)
    if verbose:
        print("".join(logs))
    return lib


if __name__ == "__main__":
    import sys
    print(build_calls(force="--force" in sys.argv))
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug_bounds="--debug-bounds" in sys.argv))
