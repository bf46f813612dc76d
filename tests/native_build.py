"""Compiles host C++ of tests/native together with sources of the library into a shared object."""
import ctypes
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_09932_gb300", "csrc")


def cuda_include():
    for home in (os.environ.get("CUDA_HOME"), "/usr/local/cuda",
                 os.path.dirname(os.path.dirname(shutil.which("nvcc") or ""))):
        if home and os.path.exists(os.path.join(home, "include", "cuda_runtime.h")):
            return os.path.join(home, "include")
    raise RuntimeError("CUDA headers not found")


def load(out_dir, name, library_sources=()):
    """tests/native/<name>.cpp and the named files of csrc/ as a ctypes library."""
    srcs = [os.path.join(ROOT, "tests", "native", name + ".cpp")]
    srcs += [os.path.join(CSRC, f) for f in library_sources]
    out = os.path.join(str(out_dir), f"lib{name}.so")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-pthread",
                        "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I", cuda_include(),
                        *srcs, "-o", out], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(r.stderr)
    return ctypes.CDLL(out)
