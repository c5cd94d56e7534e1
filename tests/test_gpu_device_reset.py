"""A flow made after the device was reset: nothing about a launch may be remembered from the
context before.  cudaDeviceReset ends a context of its own, so it runs in a child process."""
import os
import subprocess
import sys

import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes as C
import numpy as np
from paper_2208_08903_gb300 import _abi
lib = _abi.load()
rt = C.CDLL("libcudart.so.13")           # the copy the library is linked with
B, sh = 5, _abi.FlowShapeC(3, 8, 2, 32, 32, 3, 1, 0.01)   # a plan of more than 48 KB

def run():
    V, h, phi, logq = 512, C.c_void_p(), C.c_void_p(), C.c_void_p()
    w = np.random.default_rng(0).uniform(-0.05, 0.05, 1 << 17)
    _abi.check("create", lib.gf_flow_create(C.byref(sh), w.ctypes.data, _abi.GF_PREC_FP32, None, C.byref(h)))
    assert lib.gf_flow_n_params(h) <= w.size
    assert rt.cudaMalloc(C.byref(phi), C.c_size_t(4 * B * V)) == 0 and rt.cudaMalloc(C.byref(logq), C.c_size_t(8 * B)) == 0
    _abi.check("sample", lib.gf_flow_sample(h, None, B, 1, 0, None, None, phi, logq, None, None, None))
    out = np.empty(B * V, np.float32), np.empty(B)
    for o, d in zip(out, (phi, logq)):
        assert rt.cudaMemcpy(C.c_void_p(o.ctypes.data), d, C.c_size_t(o.nbytes), 2) == 0
    assert lib.gf_flow_destroy(h) == 0 and rt.cudaFree(phi) == 0 and rt.cudaFree(logq) == 0
    return out

a = run()
assert rt.cudaDeviceReset() == 0
b = run()
assert all((x == y).all() for x, y in zip(a, b)) and np.isfinite(a[1]).all()
print("ok")
"""


def test_flow_after_a_device_reset():
    require_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[-2000:]
