"""Builds libspeckv.so (sm_100a) in-tree with nvcc.  `python -m paper_2605_02888_b200.build`."""
from __future__ import annotations

import os
import subprocess
import sys

_PKG = os.path.dirname(os.path.abspath(__file__))
_CSRC = os.path.join(_PKG, "csrc")
_INC = os.path.join(os.path.dirname(_PKG), "include")
LIB_PATH = os.path.join(_CSRC, "libspeckv.so")
_SOURCES = ["speckv.cu"]
_DEPS = ["speckv.cu", "speckv_kernels.cuh", "speckv_draw.cuh", "speckv_sweep.cuh", "speckv_shard.cuh", "speckv_sample.cuh"]

NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "-shared"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


DEBUG_LIB_PATH = os.path.join(_CSRC, "libspeckv_debug.so")


def is_stale(path: str = LIB_PATH) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    deps = [os.path.join(_CSRC, d) for d in _DEPS] + [os.path.join(_INC, h) for h in ("speckv.h", "speckv_internal.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile the library if it is missing or older than its sources; return its path.
    debug=True builds the bounds-checked variant (-DSPECKV_DEBUG) beside it: every logit load and
    workspace access is compared with the call's extents, skipped and counted when outside."""
    out = DEBUG_LIB_PATH if debug else LIB_PATH
    if not force and not is_stale(out):
        return out
    tmp = out + f".tmp{os.getpid()}"
    cmd = [_nvcc(), *NVCC_FLAGS, *(["-DSPECKV_DEBUG"] if debug else []), "-I", _INC, "-o", tmp] + [os.path.join(_CSRC, s) for s in _SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), file=sys.stderr)
    subprocess.check_call(cmd)
    os.replace(tmp, out)
    return out


def torch_lib_path() -> str:
    """Where the native argument marshalling built for this Python and this torch lies.  It reads torch's C++ objects directly, so
    one built for another torch must not be loaded, and the name says which one it is for."""
    import sysconfig

    import torch
    tag = f"torch{torch.__version__}.{sysconfig.get_config_var('SOABI')}.abi{int(torch.compiled_with_cxx11_abi())}"
    return os.path.join(_CSRC, "_speckv_torch." + "".join(c if c.isalnum() or c in ".-" else "_" for c in tag) + ".so")


def build_torch(force: bool = False) -> str:
    """Compile the native argument marshalling (csrc/speckv_torch.cpp, host code only) against the installed torch if it is
    missing or older than its sources; return its path."""
    deps = [os.path.join(_CSRC, "speckv_torch.cpp"), os.path.join(_INC, "speckv.h")]
    out = torch_lib_path()
    if not force and os.path.exists(out) and all(os.path.getmtime(d) <= os.path.getmtime(out) for d in deps):
        return out
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.sep in _nvcc() else "/usr/local/cuda"
    inc = [*cpp_extension.include_paths(), sysconfig.get_paths()["include"], os.path.join(cuda, "include"), _INC]
    tmp = out + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", *(a for d in inc for a in ("-isystem", d)),
           "-o", tmp, deps[0], *(f"-L{d}" for d in cpp_extension.library_paths()), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.check_call(cmd)
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    build_torch(force="--force" in sys.argv)
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
