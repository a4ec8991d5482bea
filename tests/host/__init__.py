"""Builds the C++ harnesses of this folder: the kernels' host-callable
arithmetic (``paper_2311_17174_gb300/csrc/*.cuh``) compiled with the host
compiler, for tests without a GPU."""
import ctypes
import functools
import os
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_2311_17174_gb300", "csrc")


@functools.cache
def load(name):
    """The harness ``name``.cpp as a ctypes library."""
    inc = next((p for p in (os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                            "/usr/local/cuda/include") if os.path.exists(os.path.join(p, "cuda_runtime.h"))), None)
    if inc is None:
        pytest.skip("no CUDA headers")
    out = os.path.join(tempfile.mkdtemp(prefix="emri_host_"), name + ".so")
    # -Bsymbolic: a harness's own fakes, not the CUDA runtime that torch has loaded
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC,
                        "-I", inc, os.path.join(HERE, name + ".cpp"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)
