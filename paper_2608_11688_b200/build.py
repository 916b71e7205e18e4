"""Builds libapex.so (sm_100a) in-tree with nvcc.  Cross-compiles without a GPU."""
from __future__ import annotations

import os
import platform
import subprocess
import sys
import sysconfig
import warnings
from typing import Optional

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libapex.so")
# (named for the interpreter it is built for: another Python version builds and loads its own)
PYCALL = os.path.join(HERE, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))  # argument marshalling of the Python binding (csrc/pycall.c)
TRACE_LIB = os.path.join(HERE, "libapex_trace.so")   # the same sources with the kernels' time stamps compiled in (trace.py)
SOURCES = ["apex_ctx.cu", "apex_step.cu", "apex_observe.cu", "apex_decode.cu", "kernels_decode.cu", "kernels_decode_tiles.cu", "kernels_router.cu", "kernels_ffn.cu", "kernels_plan.cu", "kernels_ffn_tc.cu", "apex_noalloc.cu", "fit_cdf.cu", "distill.cu", "workspace.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.isabs(c) and os.path.exists(c) or not os.path.isabs(c)):
            return c
    return "nvcc"


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".hpp"))] + [os.path.join(HERE, "..", "include", "apex.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_pycall(force: bool = False) -> Optional[str]:
    """The binding's extension module (C, CPython API).  It is an accelerator: where it cannot be built (a host other than
    x86-64, no C compiler, no Python headers) None is returned and the binding marshals through ctypes."""
    if platform.machine().lower() not in ("x86_64", "amd64"):
        return None
    src = os.path.join(CSRC, "pycall.c")
    if not force and os.path.exists(PYCALL) and os.path.getmtime(src) <= os.path.getmtime(PYCALL):
        return PYCALL
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"], src, "-o", PYCALL]
    try:
        r = subprocess.run(cmd, capture_output=True, text=True)
        why = (r.stdout + r.stderr).strip() if r.returncode != 0 else None
    except OSError as e:
        why = str(e)
    if why is None:
        return PYCALL
    if os.path.exists(PYCALL):   # built from an older source
        os.remove(PYCALL)
    warnings.warn(f"csrc/pycall.c was not built, the binding goes through ctypes: {why}", RuntimeWarning)
    return None


def build(force: bool = False, verbose: bool = False) -> str:
    """Compiles every .cu of the package for sm_100a and links libapex.so (and builds the binding's extension module).
    Returns its path."""
    build_pycall(force)
    if not force and not _stale():
        return LIB
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
    if verbose:
        flags += ["-Xptxas", "-v"]
    objs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc()] + flags + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        objs.append(obj)
    cmd = [_nvcc(), "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("link failed")
    return LIB


def build_trace(force: bool = False) -> str:
    """libapex_trace.so: every kernel records (kernel id, start, end) of its first block in a device-side log, and the
    expert-FFN kernels per-CTA phase stamps (-DAPEX_TIMELINE).  The log is shared by all translation units, hence
    relocatable device code and one nvcc invocation.  Used by trace.py only; the product library carries no stamps."""
    if not force and not _stale(TRACE_LIB):
        return TRACE_LIB
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")] + ["-DAPEX_TIMELINE", "-rdc=true"]
    cmd = [_nvcc()] + flags + ["-shared", "-o", TRACE_LIB] + [os.path.join(CSRC, f) for f in SOURCES]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("nvcc failed on the trace build")
    return TRACE_LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    if "--trace" in sys.argv:
        print(build_trace(force="--force" in sys.argv))
