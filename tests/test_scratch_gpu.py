"""Scratch blocks kept between single-step calls: contexts, threads, and what gives them back."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Gram matrices in the device's primary context, in a second context, and in the first again, one call each, with memory of
# the context that is current: a block kept from the first context may not be used in the second. Small integers, so exact.
TWO_CONTEXTS = r"""
import ctypes as C, sys
import numpy as np
sys.path.insert(0, %r)
import paper_1701_03989_gb300 as P
cu = C.CDLL("libcuda.so.1")
def ok(r): assert r == 0, r
ok(cu.cuInit(0))
dev, one, two = C.c_int(), C.c_void_p(), C.c_void_p()
ok(cu.cuDeviceGet(C.byref(dev), 0))
ok(cu.cuDevicePrimaryCtxRetain(C.byref(one), dev))
ok(cu.cuCtxCreate_v2(C.byref(two), 0, dev))
Y = np.random.default_rng(0).integers(-8, 9, (5, 1000)).astype(np.float64)
def gram(ctx):
    ok(cu.cuCtxSetCurrent(ctx))
    y, g, out = C.c_uint64(), C.c_uint64(), np.zeros((5, 5))
    ok(cu.cuMemAlloc_v2(C.byref(y), C.c_size_t(Y.nbytes))); ok(cu.cuMemAlloc_v2(C.byref(g), C.c_size_t(200)))
    ok(cu.cuMemcpyHtoD_v2(y, C.c_void_p(Y.ctypes.data), C.c_size_t(Y.nbytes)))
    P.ascg_gram(1000, 5, y.value, 1000, g.value)
    ok(cu.cuMemcpyDtoH_v2(C.c_void_p(out.ctypes.data), g, C.c_size_t(200)))
    return out
for ctx in (one, two, one, two):
    assert np.array_equal(gram(ctx), Y @ Y.T)
print("ok")
"""


def test_blocks_stay_in_their_context():
    r = subprocess.run([sys.executable, "-c", TWO_CONTEXTS % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
