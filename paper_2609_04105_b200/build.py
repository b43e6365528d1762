"""Builds, in-tree, the C-ABI shared library (libfp4attn.so, nvcc for sm_100a) and the binding's native marshalling module
(_fp4attn_native.<Python's ABI tag>.torch-<version>.so, C++ against the installed torch)."""
from __future__ import annotations

import importlib.metadata
import importlib.util
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfp4attn.so")
SOURCES = ["api.cu", "quantize.cu", "attn_fwd.cu", "attn_fwd_2q.cu", "attn_fwd_fp8pv.cu", "probes.cu"]
FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
         "-Xcompiler", "-fPIC", "--shared", "-Xptxas", "-v", "--threads", "4"]


def native_path() -> str:
    """Where the marshalling module for the running Python and the installed torch belongs.  It uses torch's C++ classes, so one
    that was built against another version must neither be loaded nor pass for up to date."""
    tag = f"{sysconfig.get_config_var('SOABI')}.torch-{importlib.metadata.version('torch')}"
    return os.path.join(HERE, f"_fp4attn_native.{tag}.so")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _run(cmd, verbose: bool, target: str) -> str:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed building {os.path.basename(target)}")
    return res.stderr


def _build_native(target: str, verbose: bool) -> None:
    torch_dir = os.path.dirname(importlib.util.find_spec("torch").origin)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [sysconfig.get_paths()["include"], os.path.join(torch_dir, "include"),
               os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), os.path.join(cuda, "include")]
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-DNDEBUG"] +
         [f"-I{d}" for d in include] + [os.path.join(CSRC, "native.cpp"), "-o", target, f"-L{os.path.join(torch_dir, 'lib')}",
                                        "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"], verbose, target)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into one shared library, and the marshalling module; returns the library's path."""
    header = os.path.join(HERE, "..", "include", "fp4attn.h")
    if force or _stale(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [header]):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        log = _run([nvcc] + FLAGS + [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB], verbose, LIB)
        with open(os.path.join(HERE, "ptxas_info.txt"), "w") as f:
            f.write(log)
    native = native_path()
    if force or _stale(native, [os.path.join(CSRC, "native.cpp"), header]):
        _build_native(native, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
