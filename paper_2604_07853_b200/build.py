"""Build libqarl.so (the C-ABI CUDA library, nvcc for sm_100a) and _native.so (the Python marshalling of its
hot calls, against torch's headers) in-tree."""
from __future__ import annotations

import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libqarl.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_KEY = os.path.join(HERE, "_native.key")  # what _native.so was built against
SOURCES = ["api.cu", "quantize.cu", "permute.cu", "combine.cu", "gemm_sm100.cu", "gemm_decode_sm100.cu", "harness.cu", "linear_static.cu",
           "gemm_w4a16_sm100.cu", "api_ext.cu", "api_ep.cu", "gemm_bf16_sm100.cu", "tbpo.cu", "router.cu", "router_fused_sm100.cu", "router_cluster_sm100.cu", "moe_bwd.cu"]
HEADERS = ["common.cuh", "quant_device.cuh", "w4_dequant.cuh", "ptx_sm100.cuh", "sched.cuh", "router_select.cuh", "api_util.cuh", os.path.join("..", "..", "include", "qarl.h"),
           os.path.join("..", "..", "include", "qarl_harness.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static",
]


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in sources] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def native_key() -> str:
    """The interpreter and the torch whose headers and libraries _native.so depends on: built against others it may fail to
    import, or import and misread their objects."""
    import importlib.metadata
    import importlib.util
    import sysconfig

    where = os.path.dirname(importlib.util.find_spec("torch").origin)
    return "\n".join((sysconfig.get_config_var("SOABI"), sysconfig.get_paths()["include"], importlib.metadata.version("torch"), where))


def _native_is_for_this_python() -> bool:
    try:
        with open(NATIVE_KEY) as f:
            return f.read() == native_key()
    except OSError:
        return False


def _build_native() -> None:
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    subprocess.check_call([
        os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", os.path.join(CSRC, "native_binding.cpp"),
        "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
        "-I" + sysconfig.get_paths()["include"], "-I/usr/local/cuda/include", "-o", tmp, "-L" + HERE, "-l:libqarl.so",
        "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10",
        "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, NATIVE)
    with open(NATIVE_KEY, "w") as f:
        f.write(native_key())


def _build_library(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, *NVCC_FLAGS]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, f) for f in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is missing or older than its sources; returns the library's path."""
    if force or _stale(LIB, SOURCES + HEADERS):
        _build_library(verbose)
    if (force or not _native_is_for_this_python() or
            _stale(NATIVE, ["native_binding.cpp", os.path.join("..", "..", "include", "qarl.h")])):
        _build_native()
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
