"""Builds libcunbody.so in-tree with nvcc for sm_103a (GB300).

Each ``csrc/*.cu`` translation unit is compiled in parallel into
``_build/``; the objects are linked into ``libcunbody.so`` next to this
file (the CUDA runtime is linked statically, so the library loads without
a CUDA runtime on the library path). Rebuilds only when a source or
header is newer than the library. ``csrc/cn_binding.cpp``, the native part of
the Python binding, is compiled beside it against the installed PyTorch;
where that cannot be done the binding marshals in Python.
"""

from __future__ import annotations

import concurrent.futures as cf
import glob
import importlib.util
import os
import re
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libcunbody.so")
# debug variant: every schedule index checked on the device (CN_DEBUG_BOUNDS)
DEBUG_BUILD_DIR = os.path.join(HERE, "_build_debug")
DEBUG_LIB = os.path.join(HERE, "libcunbody_debug.so")
BINDING_SRC = os.path.join(CSRC, "cn_binding.cpp")
BINDING = os.path.join(HERE, "_binding.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-ftz=true", "-Xcompiler", "-fPIC,-O2,-fvisibility=hidden",
              "-I", INCLUDE, "-I", CSRC]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA 13 toolkit is required to build libcunbody")


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newest_input() -> float:
    files = _sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h"))
    files += glob.glob(os.path.join(INCLUDE, "*.h")) + [os.path.abspath(__file__)]
    return max(os.path.getmtime(f) for f in files)


def _compile(src: str, verbose: bool, debug_bounds: bool = False) -> str:
    obj = os.path.join(DEBUG_BUILD_DIR if debug_bounds else BUILD_DIR, os.path.basename(src)[:-3] + ".o")
    cmd = [nvcc(), *ARCH, *NVCC_FLAGS, *(["-DCN_DEBUG_BOUNDS"] if debug_bounds else []), "-c", src, "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc failed for {os.path.basename(src)}:\n{res.stderr}")
    if verbose and res.stderr:
        print(res.stderr)
    return obj


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """Compile and link libcunbody.so (or, with debug_bounds, the checked
    variant libcunbody_debug.so); returns its path."""
    lib = DEBUG_LIB if debug_bounds else LIB
    if not force and os.path.exists(lib) and os.path.getmtime(lib) >= _newest_input():
        return lib
    os.makedirs(DEBUG_BUILD_DIR if debug_bounds else BUILD_DIR, exist_ok=True)
    srcs = _sources()
    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(srcs), os.cpu_count() or 1))) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose, debug_bounds), srcs))
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"nvcc link failed:\n{res.stderr}")
    os.replace(tmp, lib)
    return lib


def build_binding(force: bool = False):
    """Compile _binding.so against the installed PyTorch (nothing of it is
    imported); returns its path, or None where that cannot be done."""
    spec = importlib.util.find_spec("torch")
    if spec is None or not spec.submodule_search_locations:
        return None
    home = spec.submodule_search_locations[0]
    try:
        with open(os.path.join(home, "version.py")) as f:
            version = re.search(r"__version__ = ['\"]([^'\"]+)", f.read()).group(1)
        inputs = [BINDING_SRC, os.path.abspath(__file__), os.path.join(home, "version.py")]
        if not force and os.path.exists(BINDING) and os.path.getmtime(BINDING) >= max(map(os.path.getmtime, inputs)):
            return BINDING
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
        tmp = BINDING + f".tmp{os.getpid()}"
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-w",
               f'-DCN_TORCH_VERSION="{version}"', "-I", sysconfig.get_paths()["include"],
               "-I", os.path.join(home, "include"), "-I", cuda, BINDING_SRC, "-o", tmp,
               "-L", os.path.join(home, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(res.stderr[-2000:])
        os.replace(tmp, BINDING)
        return BINDING
    except (OSError, AttributeError, RuntimeError) as e:
        print(f"the native part of the Python binding was not built: {e}", file=sys.stderr)
        return None


if __name__ == "__main__":
    build_binding(force=True)
    print(build(force=True, verbose=True))
