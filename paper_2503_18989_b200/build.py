"""Builds the C-ABI CUDA library (libhat.so) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import glob
import os
import shlex
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhat.so")
CALLS_SRC = os.path.join(CSRC, "calls.c")
# the binding's calls as a CPython extension, named for the interpreter it is built for; without it ctypes makes them
CALLS = os.path.join(HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC",
    "--expt-relaxed-constexpr",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the CUDA library cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


HAT_H = os.path.join(HERE, "..", "include", "hat.h")


def is_stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [HAT_H])


def build_calls(force: bool = False) -> None:
    """The extension, where this interpreter's headers are installed."""
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")):
        print(f"no Python.h in {include}: the binding's calls stay with ctypes", file=sys.stderr)
    elif force or _older(CALLS, [CALLS_SRC, HAT_H]):
        tmp = CALLS + f".tmp{os.getpid()}"
        subprocess.check_call([*shlex.split(os.environ.get("CC") or "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", include, CALLS_SRC, "-o", tmp])
        os.replace(tmp, CALLS)


LIB_DEBUG = os.path.join(HERE, "libhat_debug.so")


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library; returns its path.
    debug=True builds libhat_debug.so with -DHAT_DEBUG_BOUNDS: device-side range checks of block-table lookups, page
    ids, ring slots, TMEM columns and output rows that report through the plan's status word instead of trapping
    (load it with HAT_LIB=debug)."""
    build_calls(force)
    if debug:
        return _build(LIB_DEBUG, "_build_debug", ["-DHAT_DEBUG_BOUNDS"], verbose)
    if not force and not is_stale():
        return LIB
    return _build(LIB, "_build", [], verbose)


def _build(lib: str, obj_name: str, extra, verbose: bool) -> str:
    objs = []
    obj_dir = os.path.join(HERE, obj_name)
    os.makedirs(obj_dir, exist_ok=True)
    procs = []
    for src in sources():
        obj = os.path.join(obj_dir, os.path.basename(src)[:-3] + ".o")
        cmd = [_nvcc(), *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip() and (verbose or p.returncode != 0):
            print(out, file=sys.stderr)
        if p.returncode != 0:
            failed = True
            print(f"nvcc failed on {src}", file=sys.stderr)
    if failed:
        raise RuntimeError("CUDA build failed")
    tmp = lib + f".tmp{os.getpid()}"
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-lcudart_static", "-ldl", "-lpthread", "-lrt"])
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
