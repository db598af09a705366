"""Builds paper_2604_11288_b200/libta.so from csrc/*.cu with nvcc for sm_100a (cross-compiles without a GPU), and the CPython
module _ta_call (argument marshalling of the most frequent calls, for the Python that runs this) from csrc/py_call.cpp with g++.
The module saves host time and nothing depends on it: where it cannot be built (no Python headers, no C++ compiler) those calls
go through ctypes like the others."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB_PATH = os.path.join(_HERE, "libta.so")
CALL_PATH = os.path.join(_HERE, "_ta_call" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
CALL_SOURCE = os.path.join(_HERE, "csrc", "py_call.cpp")


def sources():
    return sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))


def headers():
    return glob.glob(os.path.join(_HERE, "csrc", "*.cuh")) + glob.glob(os.path.join(_HERE, "csrc", "*.h")) + glob.glob(
        os.path.join(_ROOT, "include", "*.h"))


def _stale():
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(d) > t for d in sources() + headers())


def _build_call(force: bool) -> None:
    header = os.path.join(_ROOT, "include", "ta.h")
    if not force and os.path.exists(CALL_PATH) and all(os.path.getmtime(f) <= os.path.getmtime(CALL_PATH)
                                                       for f in (CALL_SOURCE, header)):
        return
    try:
        subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-I",
                        os.path.join(_ROOT, "include"), "-I", sysconfig.get_paths()["include"], CALL_SOURCE, "-o",
                        CALL_PATH], check=True, capture_output=True, text=True)
    except (OSError, subprocess.CalledProcessError) as e:
        if os.path.exists(CALL_PATH):  # older than the source or the header
            os.remove(CALL_PATH)
        print(f"_ta_call was not built, its calls go through ctypes: {e}\n{getattr(e, 'stderr', None) or ''}", file=sys.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into one shared library, and the marshalling module. Returns the library's path."""
    _build_call(force)
    if not force and not _stale():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    build_dir = os.path.join(_HERE, "_build")
    os.makedirs(build_dir, exist_ok=True)
    common = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(_ROOT, "include"), "-I", os.path.join(_HERE, "csrc")]
    if verbose:
        common += ["-Xptxas", "-v"]
    procs = []
    for src in sources():
        obj = os.path.join(build_dir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        procs.append((src, subprocess.Popen(common + ["-c", src, "-o", obj], stdout=subprocess.PIPE,
                                            stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip():
            print(out, file=sys.stderr)
        if p.returncode != 0:
            failed = True
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.run([nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB_PATH] + objs +
                   ["-cudart", "static", "-ldl"], check=True)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
