"""Compile the CUDA library (nvcc, sm_100a) and the native call layer (g++, against torch) in-tree; works without a GPU."""
import os
import subprocess
import sys
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgproj_attn.so")
CALLS_SOURCE = os.path.join(CSRC, "torch_calls.cpp")
SOURCES = [os.path.join(CSRC, "gproj_attn.cu")]
ABI_HEADER = os.path.join(ROOT, "include", "gproj_attn.h")
HEADERS = [os.path.join(CSRC, f) for f in ("host_rules.h", "tile_schedule.h", "wait_budget.h", "sm100_primitives.cuh", "attn_fwd.cuh", "attn_fwd_w64.cuh", "attn_bwd.cuh", "attn_bwd_w128.cuh", "key_smoothing.cuh", "attn_fp32.cuh")] + \
          [ABI_HEADER]


def calls_path() -> str:
    """The native call layer of this Python and this torch: it is bound to the binary interfaces of both, so each pair has its own file."""
    import torch

    return os.path.join(PKG, f"_torch_calls.{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def nvcc_command(verbose: bool = False):
    cmd = ["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + SOURCES
    if verbose:
        cmd[1:1] = ["-Xptxas", "-v"]
    return cmd


def calls_command():
    import sysconfig

    import torch
    from torch.utils.cpp_extension import CUDA_HOME, include_paths, library_paths

    includes = [os.path.dirname(ABI_HEADER)] + include_paths() + [sysconfig.get_paths()["include"], os.path.join(CUDA_HOME or "/usr/local/cuda", "include")]
    return ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] + \
        [f"-I{p}" for p in includes] + ["-o", calls_path(), CALLS_SOURCE] + [f"-L{p}" for p in library_paths()] + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]


def _up_to_date(target, deps):
    return os.path.exists(target) and all(os.path.getmtime(target) >= os.path.getmtime(p) for p in deps)


def _run(cmd, verbose=False):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed:\n" + res.stdout + res.stderr)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or not _up_to_date(LIB, SOURCES + HEADERS):
        _run(nvcc_command(verbose), verbose)
    if force or not _up_to_date(calls_path(), [CALLS_SOURCE, ABI_HEADER]):
        try:                       # optional: without it the calls go through ctypes
            _run(calls_command())
        except (OSError, RuntimeError) as e:
            if os.path.exists(calls_path()):
                os.remove(calls_path())                     # out of date: it may call the library by another signature
            warnings.warn(f"the native call layer was not built, so calls take more host time: {e}", RuntimeWarning, stacklevel=2)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
