"""Host-compilable parts of the device headers as a shared library for CPU tests: the same source text, its
single-precision operations left uncontracted (the library's own flags do that on the device)."""

import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_02150_gb300", "csrc")


def compile_host(source, folder):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, lib = os.path.join(folder, "host_code.cu"), os.path.join(folder, "host_code.so")
    with open(src, "w") as f:
        f.write(source)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC,-ffp-contract=off", "-gencode",
                        "arch=compute_103a,code=sm_103a", "-I", CSRC, "-shared", "-o", lib, src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(lib)
