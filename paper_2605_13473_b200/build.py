"""Builds the CUDA library in-tree with nvcc for sm_100a (no GPU needed)."""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libosdn.so")
# python module: argument marshalling of the hot calls.  Its name carries the interpreter's ABI, so that another one does
# not load it.
CALL_LIB = os.path.join(HERE, "_osdn_call" + sysconfig.get_config_var("EXT_SUFFIX"))
SOURCES = ["osdn_api.cu", "osdn_phase1.cu", "osdn_simt.cu", "osdn_tc.cu", "osdn_decode.cu", "osdn_kda.cu"]


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def _torch_dir() -> str:
    return os.path.dirname(importlib.util.find_spec("torch").origin)


def call_inputs() -> list:
    """What the extension module is built from; torch's C++ interface changes with its version."""
    return [os.path.join(CSRC, "call.cpp"), os.path.join(os.path.dirname(HERE), "include", "osdn.h"),
            os.path.join(_torch_dir(), "version.py")]


def _build_call(force: bool) -> None:
    if not force and os.path.exists(CALL_LIB) and os.path.getmtime(CALL_LIB) >= _newest(call_inputs()):
        return
    src, torch_dir = call_inputs()[0], _torch_dir()
    inc = os.path.join(torch_dir, "include")
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden", "-I" + inc,
                    "-I" + os.path.join(inc, "torch", "csrc", "api", "include"), "-I/usr/local/cuda/include",
                    "-I" + sysconfig.get_paths()["include"], "-o", CALL_LIB, src, "-L" + HERE, "-l:libosdn.so",
                    "-L" + os.path.join(torch_dir, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                    "-Wl,-rpath,$ORIGIN"], check=True)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    deps = srcs + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "osdn.h"))
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest(deps):
        _build_call(False)
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "--threads", "0", "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-Xcompiler", "-fPIC", "-shared", "-o", LIB] + srcs
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    _build_call(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
