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


# A program that never creates an operator: what its calls keep comes back by ascg_trim, and they go on working.
NO_OPERATOR = r"""
import sys
import torch
sys.path.insert(0, %r)
import paper_1701_03989_gb300 as P
Y = torch.rand((5, 2048), dtype=torch.float64, device="cuda")
G = torch.empty((5, 5), dtype=torch.float64, device="cuda")
def gram():
    P.ascg_gram(2048, 5, Y, 2048, G)
    return G.cpu()  # compared on the host: torch's own kernels would load, and take device memory, on first use
first = gram()
P.ascg_trim()
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for _ in range(3):
    assert torch.equal(gram(), first)
    P.ascg_trim()
assert torch.cuda.mem_get_info()[0] == free
print("ok")
"""


def test_trim_without_an_operator():
    r = subprocess.run([sys.executable, "-c", NO_OPERATOR % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


def test_trim_gives_an_operators_workspace_back():
    """Matrix powers keep at most the folded operator that the header states; trimming gives it back and changes no bit."""
    import paper_1701_03989_gb300 as P

    n, s = 1 << 20, 16  # tridiagonal: O has two entries a row
    cols = np.arange(n)[:, None] + np.array([-1, 0, 1])[None, :]
    keep = (cols >= 0) & (cols < n)
    vals = np.broadcast_to(np.array([-1.0, 4.0, -1.0]), (n, 3))
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    op = P.ascg_op_create_csr(n, int(rowptr[-1]), rowptr, cols[keep].astype(np.int32), vals[keep], 0)
    th, sg, gm = np.linspace(0.5, 3.5, s), np.full(s, 0.25), np.array([1.0] + [0.5] * (s - 1))
    Y = torch.zeros((2 * s + 1, n), dtype=torch.float64, device="cuda")
    Y[:2] = torch.rand((2, n), dtype=torch.float64, device="cuda")
    P.ascg_matrix_powers(op, s, th, sg, gm, Y, n)
    want = Y.cpu()
    torch.cuda.synchronize()
    P.ascg_trim(op)
    free = torch.cuda.mem_get_info()[0]
    P.ascg_matrix_powers(op, s, th, sg, gm, Y, n)
    kept = free - torch.cuda.mem_get_info()[0]
    assert 0 < kept <= 8 * n * s + 8 * 2 * n + (4 << 20)  # one gamma other than 1; allocations come in 2 MB
    assert torch.equal(Y.cpu(), want)
    P.ascg_trim(op)
    assert torch.cuda.mem_get_info()[0] == free
    b, x = torch.rand(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    assert P.ascg_solve(op, b, x, P.make_options(s_max=4)).status == P.ASCG_OK
    P.ascg_op_destroy(op)


def test_mixed_calls_from_threads():
    """Calls that stage through the pinned page, on a stream each: every one of them runs, with the bits it has alone."""
    import paper_1701_03989_gb300 as P

    n, w, s = 4096, 17, 8
    g = torch.Generator(device="cuda").manual_seed(1)
    Y = torch.rand((w, n), dtype=torch.float64, device="cuda", generator=g) - 0.5
    G0 = (Y @ Y.T).contiguous()
    coords = torch.rand(3 * w, dtype=torch.float64, device="cuda", generator=g)
    rng = np.random.default_rng(2)

    def gram(k, st):
        G = torch.empty((w, w), dtype=torch.float64, device="cuda")
        P.ascg_gram(n, w, Y, n, G, stream=st)
        return G.cpu().numpy()

    def block(k, st):
        c = torch.zeros(3 * w, dtype=torch.float64, device="cuda")
        info, hist = P.ascg_block_step(s, G0, P.ASCG_ADAPTIVE, np.full(s, 0.1 * k), np.zeros(s), np.ones(s), n, 1e-9, 1.0,
                                       1, 100, 1.0, c, stream=st)
        return np.concatenate([np.array(info.sqrt_kappa), hist.ravel(), c.cpu().numpy()])

    al, be = rng.uniform(0.3, 3.0, (8, 16)), rng.uniform(0.01, 1.5, (8, 15))

    def shifts(k, st):
        return P.ascg_newton_shifts(al[k], be[k], 16, 16, stream=st)

    def recover(k, st):
        v = torch.zeros((3, n), dtype=torch.float64, device="cuda")
        P.ascg_recover_tc(n, w, Y, n, coords, v[0], v[1], v[2], stream=st)
        return v.cpu().numpy()

    calls = [gram, block, shifts, recover]
    alone = {(f, k): f(k, None) for f in calls for k in range(8)}
    done, errors = [0] * 8, []

    def work(k):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for i in range(40):
                    f = calls[(k + i) % 4]
                    assert np.array_equal(f(k, st), alone[f, k]), (f, k)
                    done[k] += 1
        except BaseException as e:  # a thread's failure is the test's
            errors.append((k, repr(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors and done == [40] * 8
