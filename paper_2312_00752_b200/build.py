"""Compiles the CUDA sources in csrc/ into libssm_scan.so next to this file (sm_100a only, in-tree), and the binding's
argument marshalling (csrc/marshal.cpp, against torch's headers) into _marshal-<torch>-<python>.so."""
from __future__ import annotations

import glob
import importlib.util
import os
import shutil
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")
LIB_PATH = os.path.join(_HERE, "libssm_scan.so")
# the same library with every tile / global index of the tuned kernels range-checked (-DSSM_DEBUG_BOUNDS)
DEBUG_LIB_PATH = os.path.join(_HERE, "libssm_scan_debug.so")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "-cudart", "static"]

MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build_library(force: bool = False, verbose: bool = False, extra_flags=(), debug_bounds: bool = False) -> str:
    """nvcc -shared of every .cu file; returns the path of the library.  Raises if nvcc fails.  With debug_bounds the
    bounds-checking variant is built into DEBUG_LIB_PATH instead (objects in a directory of their own)."""
    if debug_bounds:
        return _build(DEBUG_LIB_PATH, ".dbg.o", ("-DSSM_DEBUG_BOUNDS", *extra_flags), verbose)
    if not force and not is_stale():
        return LIB_PATH
    return _build(LIB_PATH, ".o", tuple(extra_flags), verbose)


def _build(lib_path: str, obj_suffix: str, extra_flags, verbose: bool) -> str:
    nvcc = os.environ.get("NVCC", "nvcc")
    objs = []
    procs = []
    for src in sources():
        obj = os.path.splitext(src)[0] + obj_suffix
        cmd = [nvcc, *NVCC_FLAGS, *extra_flags, "-I", INCLUDE, "-I", CSRC, "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            print(out)
        if pr.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = lib_path + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-shared", "-cudart", "static", *objs, "-o", tmp], check=True)
    os.replace(tmp, lib_path)
    return lib_path


if __name__ == "__main__":
    import sys
    print(build_library(force=True, verbose="-v" in sys.argv))


def marshal_path() -> str:
    """Where the marshalling module for the torch and the interpreter in use lies.  It is C++ against torch's headers and
    fits no other build of torch, which file dates do not show, so both are in its name."""
    import torch
    tag = f"torch{torch.__version__}.{(torch.version.git_version or '')[:8]}-{sysconfig.get_config_var('SOABI')}"
    return os.path.join(_HERE, f"_marshal-{tag}.so")


def marshal_is_stale() -> bool:
    path = marshal_path()
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(d) > t for d in [MARSHAL_SOURCE, *glob.glob(os.path.join(INCLUDE, "*.h"))])


def build_marshal(force: bool = False) -> str:
    """g++ -shared of the marshalling module; returns its path.  Raises if the compiler fails."""
    path = marshal_path()
    if not force and not marshal_is_stale():
        return path
    torch_dir = importlib.util.find_spec("torch").submodule_search_locations[0]
    include = os.path.join(torch_dir, "include")
    cuda = os.path.dirname(os.path.dirname(shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"))
    tmp = path + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-I", INCLUDE,
           "-I", include, "-I", os.path.join(include, "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), MARSHAL_SOURCE, "-o", tmp,
           "-L", os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10", "-ldl"]
    pr = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if pr.returncode != 0:
        print(pr.stdout)
        raise RuntimeError(f"{cmd[0]} failed on {MARSHAL_SOURCE}")
    os.replace(tmp, path)
    return path
