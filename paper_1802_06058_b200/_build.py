"""Builds the CUDA library in-tree with nvcc for sm_100a and the Python binding with g++ (no JIT cache).

Every csrc/*.cu is compiled to an object file of its own (in parallel; an object is rebuilt only when its
source, a shared header or the flags changed) and the objects are linked into libvgc.so next to this file."""
from __future__ import annotations

import concurrent.futures
import glob
import hashlib
import importlib.util
import os
import subprocess
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(os.path.dirname(PKG_DIR), "include")
LIB_PATH = os.path.join(PKG_DIR, "libvgc.so")
NATIVE_SRC = os.path.join(CSRC, "vgc_binding.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_vgc_native.so")
OBJ_DIR = os.path.join(PKG_DIR, "build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", INCLUDE]
NATIVE_FLAGS = ["-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return sorted(glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h")))


def _newest(paths) -> float:
    return max(os.path.getmtime(p) for p in paths)


def _obj_path(src: str) -> str:
    tag = hashlib.sha1(" ".join(NVCC_FLAGS).encode()).hexdigest()[:8]
    return os.path.join(OBJ_DIR, os.path.splitext(os.path.basename(src))[0] + "." + tag + ".o")


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    return _newest(_sources() + _headers()) > os.path.getmtime(LIB_PATH)


def _compile(nvcc: str, src: str, verbose: bool) -> str:
    obj = _obj_path(src)
    if os.path.exists(obj) and os.path.getmtime(obj) >= _newest([src] + _headers()):
        return obj
    tmp = obj + ".tmp.%d" % os.getpid()
    cmd = [nvcc, *NVCC_FLAGS, "-c", "-o", tmp, src]
    if verbose:
        cmd[1:1] = ["-Xptxas", "-v"]
        print(" ".join(cmd))
    subprocess.run(cmd, check=True)
    os.replace(tmp, obj)
    return obj


def _native_tag() -> str:
    """What the extension module depends on beside its source: the interpreter, torch's version (its C++ ABI) and the flags."""
    import importlib.metadata
    return " ".join([sysconfig.get_config_var("SOABI") or "", importlib.metadata.version("torch"), *NATIVE_FLAGS])


def _build_native(force: bool) -> None:
    """The extension module that marshals the Python calls: compiled against torch's headers, linked to libvgc.so."""
    stamp = os.path.join(OBJ_DIR, "native.tag")
    if not force and os.path.exists(NATIVE_PATH) and os.path.getmtime(NATIVE_PATH) >= _newest([NATIVE_SRC] + _headers()):
        # (no stamp: the module came without its build folder, as on a machine that only runs it)
        if not os.path.exists(stamp) or open(stamp).read() == _native_tag():
            return
    torch_dir = importlib.util.find_spec("torch").submodule_search_locations[0]
    torch_inc, torch_lib = os.path.join(torch_dir, "include"), os.path.join(torch_dir, "lib")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = NATIVE_PATH + ".tmp.%d" % os.getpid()
    subprocess.run([os.environ.get("CXX", "g++"), *NATIVE_FLAGS,
                    "-I", INCLUDE, "-isystem", torch_inc, "-isystem", os.path.join(torch_inc, "torch", "csrc", "api", "include"),
                    "-isystem", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"), NATIVE_SRC, "-o", tmp,
                    "-L", torch_lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-L", PKG_DIR, "-lvgc",
                    "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + torch_lib], check=True)
    os.replace(tmp, NATIVE_PATH)
    os.makedirs(OBJ_DIR, exist_ok=True)
    with open(stamp, "w") as f:
        f.write(_native_tag())


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libvgc.so next to this file and the binding beside it; returns the library's path."""
    if not force and not _stale():
        _build_native(False)
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    if force:
        for old in glob.glob(os.path.join(OBJ_DIR, "*.o")):
            os.remove(old)
    srcs = _sources()
    with concurrent.futures.ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 1)) as pool:
        objs = list(pool.map(lambda s: _compile(nvcc, s, verbose), srcs))
    tmp = LIB_PATH + ".tmp.%d" % os.getpid()
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs], check=True)
    os.replace(tmp, LIB_PATH)
    _build_native(force)
    return LIB_PATH


PROBE_SRC = os.path.join(CSRC, "probe", "mma_rate_probe.cu")
PROBE_LIB_PATH = os.path.join(PKG_DIR, "libvgc_probe.so")


def build_probe() -> str:
    """The tensor-pipe rate probe behind `bench.py --mma-rates`: a measurement aid with a library of its own."""
    if os.path.exists(PROBE_LIB_PATH) and os.path.getmtime(PROBE_LIB_PATH) >= _newest([PROBE_SRC] + _headers()):
        return PROBE_LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = PROBE_LIB_PATH + ".tmp.%d" % os.getpid()
    subprocess.run([nvcc, *NVCC_FLAGS, "-I", CSRC, "-shared", "-o", tmp, PROBE_SRC], check=True)
    os.replace(tmp, PROBE_LIB_PATH)
    return PROBE_LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
