"""The first call of the allocation-free FFT on a device sets up its tables on
the caller's stream: work that is running on the default stream does not hold
it up.  In a process of its own, since the set-up happens once, with kernels
and static arrays loaded at start (CUDA_MODULE_LOADING=EAGER: loading them at
their first use waits for the device by itself), and without torch, whose
kernels would all be loaded too."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CHILD = """
import ctypes as C
import numpy as np
from paper_2311_17174_gb300 import emri as E
cu = C.CDLL("libcuda.so.1")
def ok(rc): assert rc == 0, rc
ctx = E.Context(0)                     # makes the device's context current
def alloc(nbytes):
    p = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(nbytes)))
    return p.value
n, N, B = 1 << 16, 1 << 20, 32
x = np.random.default_rng(1).standard_normal((n, 2)).view(np.complex128)[:, 0].copy()
z, busy = alloc(x.nbytes), alloc(N * B * 16)
ok(cu.cuMemcpyHtoD_v2(C.c_uint64(z), x.ctypes.data_as(C.c_void_p), C.c_size_t(x.nbytes)))
ok(cu.cuMemsetD32_v2(C.c_uint64(busy), 0, C.c_size_t(N * B * 4)))
s, done = C.c_void_p(), C.c_void_p()
ok(cu.cuStreamCreate(C.byref(s), 1))   # CU_STREAM_NON_BLOCKING
ok(cu.cuEventCreate(C.byref(done), 2))
ctx.fft_batch(busy, N, B, E.FP64, -1, stream=0)
ok(cu.cuCtxSynchronize())
for _ in range(400):                   # about half a second of the default stream
    ctx.fft_batch(busy, N, B, E.FP64, -1, stream=0)
ok(cu.cuEventRecord(done, None))
E.fft_batch_noalloc(z, n, 1, E.FP64, -1, stream=s.value)
assert cu.cuEventQuery(done) == 600, "the set-up waited for the default stream"   # CUDA_ERROR_NOT_READY
ok(cu.cuCtxSynchronize())
y = np.empty_like(x)
ok(cu.cuMemcpyDtoH_v2(y.ctypes.data_as(C.c_void_p), C.c_uint64(z), C.c_size_t(x.nbytes)))
ref = np.fft.fft(x)
assert np.linalg.norm(y - ref) <= 3e-15 * np.linalg.norm(ref)
print("ok")
"""


def test_setup_waits_for_its_own_stream_only():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CUDA_MODULE_LOADING="EAGER"))
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr
