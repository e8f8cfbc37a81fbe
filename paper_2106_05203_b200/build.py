"""Builds libef21.so (sm_100a, nvcc) and the Python call of its standalone Top-k (_topk_call.so, the C++ compiler, against
torch's headers) next to this file.  No GPU is needed to build."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libef21.so")
CALL = os.path.join(HERE, "_topk_call.so")
CALL_SOURCE = os.path.join(CSRC, "topk_call.cpp")


def nvcc_path() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: libef21 cannot be built")
    return cand


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _newest_source_mtime() -> float:
    files = [f for f in glob.glob(os.path.join(CSRC, "*")) if f != CALL_SOURCE] + [os.path.join(HERE, "..", "include", "ef21.h")]
    return max(os.path.getmtime(f) for f in files)


def call_built_for() -> str:
    """What _topk_call.so depends on beside its source; the module carries it as `built_for`."""
    import sysconfig
    import torch
    return f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"


def _call_is_current() -> bool:
    if not os.path.exists(CALL) or os.path.getmtime(CALL) < os.path.getmtime(CALL_SOURCE):
        return False
    with open(CALL, "rb") as f:
        return call_built_for().encode() + b"\0" in f.read()


def build_call(force: bool = False) -> str:
    if not force and _call_is_current():
        return CALL
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc_path())), "include")
    include = [sysconfig.get_paths()["include"], *cpp_extension.include_paths(), cuda]
    tmp = CALL + f".tmp{os.getpid()}"
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f'-DEF21_BUILT_FOR="{call_built_for()}"',
                    f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(f"-I{i}" for i in include), CALL_SOURCE,
                    *(f"-L{p}" for p in cpp_extension.library_paths()), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                    "-o", tmp], check=True)         # (found by name at run time: the import of torch has loaded them)
    os.replace(tmp, CALL)
    return CALL


def build(force: bool = False, verbose: bool = False) -> str:
    """Builds both; returns the path of the library."""
    build_call(force)
    return build_library(force, verbose)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compiles every csrc/*.cu to an object file (side by side: the persistent kernels of the three
    methods are translation units of their own) and links libef21.so."""
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    import tempfile
    nvcc = nvcc_path()
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC"]
    if verbose:
        flags.insert(0, "-Xptxas=-v")
    with tempfile.TemporaryDirectory(prefix="libef21_build_") as tmpdir:
        def compile_one(src: str) -> str:
            obj = os.path.join(tmpdir, os.path.basename(src) + ".o")
            cmd = [nvcc, *flags, "-c", src, "-o", obj]
            if verbose:
                print(" ".join(cmd))
            subprocess.run(cmd, check=True)
            return obj
        srcs = sources()
        with ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 1)) as pool:
            objs = list(pool.map(compile_one, srcs))
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.run([nvcc, "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                        "-o", tmp, *objs], check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
