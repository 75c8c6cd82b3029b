"""One process, several CUDA contexts of a device: kernels that need more
shared memory than a launch gets by default, and the device error word, work
in a second context and in the primary one made anew after a reset.  Each runs
as a child process that talks to the driver itself."""
import os
import subprocess
import sys

import pytest

import paper_2507_11067_gb300 as mms

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
import numpy as np
import paper_2507_11067_gb300 as mms
from paper_2507_11067_gb300 import _lib
import oracle

cu = ctypes.CDLL("libcuda.so.1")
def call(name, *a):
    assert getattr(cu, name)(*a) == 0, name
call("cuInit", 0)
ctx = ctypes.c_void_p()

def primary():
    call("cuDevicePrimaryCtxRetain", ctypes.byref(ctx), 0)
    call("cuCtxSetCurrent", ctx)

def device(a):
    p = ctypes.c_uint64()
    call("cuMemAlloc_v2", ctypes.byref(p), ctypes.c_size_t(a.nbytes))
    call("cuMemcpyHtoD_v2", p, ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(a.nbytes))
    return ctypes.c_void_p(p.value)

r, n = 2, 64
rng = np.random.default_rng(0)
grid = rng.uniform(-1, 1, (n + 4, n + 4, n + 4)).astype(np.float32)
c = rng.normal(size=125).astype(np.float32)
ref = oracle.stencil("box", r, c, grid)
lib = mms.load()

def sweeps():
    for path in (1, 4):   # CUDA cores, tensor cores (BF16x3)
        inp, out = device(grid), device(np.zeros((n, n, n), np.float32))
        d = _lib.StencilDesc(1, r, c.ctypes.data, n, n, n, 0, 0, 0, 0, path, -1)
        _lib.check(lib.mms_stencil_apply_ex(ctypes.byref(d), inp, out, None))
        _lib.check(lib.mms_check_device(None))
        got = np.empty((n, n, n), np.float32)
        call("cuMemcpyDtoH_v2", ctypes.c_void_p(got.ctypes.data), ctypes.c_uint64(out.value), ctypes.c_size_t(got.nbytes))
        err = np.abs(got - ref).max() / np.abs(ref).max()
        assert err <= 1e-5, (path, err)

def error_word():
    _lib.check(lib.mms_selftest_timeout(2000, None))
    try:
        _lib.check(lib.mms_check_device(None))
    except mms.MMSError as e:
        assert "TIMEOUT" in str(e), e
    else:
        raise AssertionError("no timeout reported")
    _lib.check(lib.mms_check_device(None))

primary()
sweeps()
error_word()
if sys.argv[1] == "second":
    call("cuCtxCreate_v2", ctypes.byref(ctx), 0, 0)
else:
    call("cuDevicePrimaryCtxReset_v2", 0)
    primary()
sweeps()
error_word()
print("ok")
"""


@pytest.mark.parametrize("how", ["second", "reset"])
def test_kernels_in_another_context(how):
    mms.build()
    r = subprocess.run([sys.executable, "-c", CHILD, how], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
