"""Compiles csrc/*.cu into libavsg.so with nvcc for sm_100a, and the binding's extension module with g++ (both in-tree)."""
import glob
import os
import subprocess
import sysconfig
import warnings

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB = os.path.join(_HERE, "libavsg.so")
CALLS_SOURCE = os.path.join(CSRC, "python_calls.cpp")
CALLS = os.path.join(_HERE, "_python_calls" + sysconfig.get_config_var("EXT_SUFFIX"))      # (of this Python)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "--use_fast_math",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(srcs) -> bool:
    if not os.path.exists(LIB):
        return True
    deps = srcs + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps)


def build_calls(force: bool = False):
    """The extension module that makes the binding's hot calls, rebuilt when a source is newer."""
    deps = [CALLS_SOURCE] + glob.glob(os.path.join(INCLUDE, "*.h"))
    if force or not os.path.exists(CALLS) or any(os.path.getmtime(d) > os.path.getmtime(CALLS) for d in deps):
        tmp = CALLS + ".tmp.%d" % os.getpid()
        subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-Wall", "-Wextra", "-Wno-missing-field-initializers",
                               "-fPIC", "-shared", "-fvisibility=hidden", "-I", sysconfig.get_paths()["include"], "-I", INCLUDE,
                               "-o", tmp, CALLS_SOURCE])
        os.replace(tmp, CALLS)
    return CALLS


def build_library(force: bool = False, verbose: bool = False):
    """Returns the path of libavsg.so, rebuilding it (and the extension module) when a source is newer.  The library needs no
    Python; where the module cannot be built (no C++ compiler, no Python.h) the binding goes without it."""
    lib = _build_library(force, verbose)
    try:
        build_calls(force)
    except (OSError, subprocess.CalledProcessError) as e:
        warnings.warn("the binding's extension module was not built (%s): calls are marshalled by ctypes" % e)
    return lib


def _build_library(force: bool, verbose: bool):
    srcs = sources()
    if not srcs:
        return None
    if force or _stale(srcs):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + ".tmp.%d" % os.getpid()
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-I", INCLUDE, "-I", CSRC,
                                                                               "-o", tmp] + srcs
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    return LIB
