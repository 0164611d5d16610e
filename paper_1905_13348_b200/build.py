"""Builds the CUDA library in-tree with nvcc for sm_100a (no GPU needed to compile), and the extension
module with the binding's per-window calls against it."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB_PATH = os.path.join(_HERE, "libinfaas_b200.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))


def calls_path() -> str:
    """The extension module for the torch and the Python that run: it looks into tensors through torch's C++
    headers, so one that was built for others is not even found."""
    import torch
    return os.path.join(_HERE, f"_calls.{sysconfig.get_config_var('SOABI')}-torch-{torch.__version__}.so")


def _stale() -> bool:
    calls = calls_path()
    if not (os.path.exists(LIB_PATH) and os.path.exists(calls)):
        return True
    deps = sources() + [os.path.join(_HERE, "csrc", "calls.cpp")] + glob.glob(os.path.join(_HERE, "csrc", "*.cuh")) + \
        glob.glob(os.path.join(_ROOT, "include", "*.h"))
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(calls))
    return any(os.path.getmtime(d) > built for d in deps)


def _build_calls() -> None:
    import torch
    top, path = os.path.dirname(torch.__file__), calls_path()
    tmp = path + f".tmp{os.getpid()}"
    subprocess.check_call(
        ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
         f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
         "-I", os.path.join(_ROOT, "include"), "-I", sysconfig.get_paths()["include"],
         "-isystem", os.path.join(top, "include"),
         os.path.join(_HERE, "csrc", "calls.cpp"), "-o", tmp,
         "-L", _HERE, "-l:libinfaas_b200.so", "-Wl,-rpath,$ORIGIN",
         "-L", os.path.join(top, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"])
    os.replace(tmp, path)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB_PATH
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(_ROOT, "include"),
           "-I", os.path.join(_HERE, "csrc")]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += sources() + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB_PATH)
    _build_calls()
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
