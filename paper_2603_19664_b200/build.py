"""Build the CUDA library in-tree: ``python -m paper_2603_19664_b200.build`` (``--check``: the checking build).

Compiles every ``csrc/*.cu`` for sm_100a with nvcc into ``libkvd.so`` next to this file.  The CUDA
runtime is linked statically and the driver API is reached through ``cudaGetDriverEntryPoint``, so
the library also loads on a machine without a GPU driver (where every entry point that needs a
device reports an error).  ``_kvdcall``, an extension module of the running interpreter, marshals the arguments of the hot
calls (csrc/kvd_pycall.c).
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkvd.so")
LIB_CHECK = os.path.join(HERE, "libkvd_check.so")  # the same sources with -DKVD_CHECK (device-side index tests)
# argument marshalling of the hot calls; named for the interpreter it is built for, which another one does not load
CALLS = os.path.join(HERE, "_kvdcall" + sysconfig.get_config_var("EXT_SUFFIX"))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
         "--expt-relaxed-constexpr"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return _sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [
        os.path.join(os.path.dirname(HERE), "include", "kvd.h")]


def needs_build(check: bool = False) -> bool:
    lib = LIB_CHECK if check else LIB
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(p) > t for p in _deps())


def build_calls(force: bool = False) -> str:
    """Compile the C half of the Python binding (gcc; no CUDA in it)."""
    src = os.path.join(CSRC, "kvd_pycall.c")
    deps = [src, os.path.join(os.path.dirname(HERE), "include", "kvd.h")]
    if force or not os.path.exists(CALLS) or any(os.path.getmtime(p) > os.path.getmtime(CALLS) for p in deps):
        tmp = CALLS + f".tmp{os.getpid()}"
        subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", tmp, src], check=True)
        os.replace(tmp, CALLS)
    untagged = os.path.join(HERE, "_kvdcall.so")  # any interpreter would load it
    if untagged != CALLS and os.path.exists(untagged):
        os.remove(untagged)
    return CALLS


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    """Compile libkvd.so, or with ``check`` libkvd_check.so: the build whose kernels test the indices they
    derive on the device and report through the status word instead of accessing out of range."""
    LIB = LIB_CHECK if check else globals()["LIB"]
    try:
        build_calls(force)
    except (OSError, subprocess.CalledProcessError) as e:  # the binding does without it: its calls then cost more host time
        sys.stderr.write(f"[build] {os.path.basename(CALLS)} not built ({e}): all calls go through ctypes\n")
    if not force and not needs_build(check):
        return LIB
    objdir = os.path.join(HERE, "build", "check") if check else os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    objs = []
    for src in _sources():
        obj = os.path.join(objdir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [NVCC, *FLAGS, *(["-DKVD_CHECK"] if check else []), "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([NVCC, "-shared", "-o", tmp, *objs, "-cudart", "static"], check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, check="--check" in sys.argv))
