"""Calls that meet the end of the memory they may allocate: the library's stream-ordered allocations come from the device's
current memory pool, and a child process puts a pool of limited size there.

A call that is refused for want of memory leaves the handle and the library as they were: the next one that fits gives the
same numbers.  The exact near rule's table per tet is an optimisation: a call that finds no room for it evaluates pair by pair, and a
table already held makes way for buffers that a later call cannot do without.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = '''
import ctypes, sys
sys.path.insert(0, %r)
import numpy as np, torch
import paper_0712_1695_gb300 as bs
from paper_0712_1695_gb300.binding import BS_ERR_CUDA, BSError
from workloads import config2_ring
torch.cuda.init()
torch.empty(1, device="cuda")
cu = ctypes.CDLL("libcuda.so.1")


class Props(ctypes.Structure):  # CUmemPoolProps: pinned device memory, no handles exported
    _fields_ = [("type", ctypes.c_int), ("handles", ctypes.c_int), ("loc", ctypes.c_int), ("dev", ctypes.c_int),
                ("sec", ctypes.c_void_p), ("max_size", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


def check(r):
    assert r == 0, r


def limit(mib):
    torch.cuda.synchronize()
    p = ctypes.c_void_p()
    check(cu.cuMemPoolCreate(ctypes.byref(p), ctypes.byref(Props(1, 0, 1, 0, None, mib << 20, 0))))
    check(cu.cuDeviceSetMemPool(0, p))


def fill():
    """Take what is left of the pool, down to pieces of 512 bytes."""
    held = []
    size = 1 << 30
    while size >= 512:
        q = ctypes.c_uint64()
        if cu.cuMemAllocAsync(ctypes.byref(q), ctypes.c_size_t(size), None) == 0:
            held.append(q)
        else:
            size >>= 1
    return held


def free(held):
    for q in held:
        check(cu.cuMemFreeAsync(q, None))


m = config2_ring(24)  # 13824 nodes, 73002 tets: a table of 68 MiB
x = torch.from_numpy(m.nodes).cuda()
few = x[::50].contiguous()
new = lambda: bs.Mesh(m.nodes, m.tets, m.omega)
EXACT = dict(far_ratio=2.0, tet_gauss_order=4, n_theta=4, n_phi=8, near_rule=bs.BS_NEAR_EXACT)


def call(h, pts, **p):
    """The velocities, or None when there was no memory for the call."""
    try:
        v = h.bs_velocity(pts, **p).cpu().numpy()
    except BSError as e:
        assert e.code == BS_ERR_CUDA, e
        return None
    h.bs_status()
    return v


def close(a, b, tol):
    return np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
'''

SCRIPTS = {
    # the error of a refused call is not met again by the next one
    "after a refused call": '''
RAY = dict(far_ratio=2.0, tet_gauss_order=64, n_theta=4, n_phi=8, precision=bs.BS_FP32)
limit(1024)
want = call(new(), few, **RAY)
limit(64)
assert call(new(), few, **RAY) is None  # 183 MiB of far records
limit(1024)
got = call(new(), few, **RAY)
assert np.array_equal(got, want)
''',
    # tables half replaced by a call that was refused are not taken for the former ones
    "refused between two calls": '''
RAY = dict(far_ratio=2.0, tet_gauss_order=4, n_theta=4, n_phi=8, precision=bs.BS_FP64)
tile = [bs.bs_variant_shape(bs.BS_FP64, 4, 0, v)["tile"] for v in range(bs.bs_num_variants(bs.BS_FP64, 4, 0))]
big, small = tile.index(32), tile.index(16)
limit(256)
h = new()
h.bs_set_variant(bs.BS_FP64, 4, 0, big)
first = call(h, few, **RAY)
h.bs_set_variant(bs.BS_FP64, 4, 0, small)
held = fill()
assert call(h, few, **RAY) is None  # twice the tile headers
h.bs_set_variant(bs.BS_FP64, 4, 0, big)
call(h, few, **RAY)
free(held)
again = call(h, few, **RAY)
assert np.array_equal(again, first)
''',
    # the table does not fit, the rest does
    "no room for the table": '''
for prec, tol in ((bs.BS_FP32, 1e-6), (bs.BS_FP64, 1e-12)):
    limit(1024)
    want = call(new(), few, precision=prec, **EXACT)
    limit(64)
    h = new()
    for _ in range(2):
        got = call(h, few, precision=prec, **EXACT)
        assert got is not None and close(got, want, tol)
    limit(1024)
    full = call(new(), x, precision=prec, **EXACT)
    limit(192)
    h = [new(), new()]
    b = bs.Batch(h)
    outs = [torch.empty_like(x), torch.empty_like(x)]
    b.bs_batch_velocity(outs, precision=prec, **EXACT)
    torch.cuda.synchronize()
    for o in outs:
        assert close(o.cpu().numpy(), full, tol)
''',
    # what a handle can do does not depend on the table it holds
    "the table makes way": '''
worked = 0
for mib in range(96, 513, 32):
    limit(mib)
    alone = call(new(), x, precision=bs.BS_FP32, **EXACT)
    limit(mib)
    h = new()
    call(h, few, precision=bs.BS_FP32, **EXACT)
    after = call(h, x, precision=bs.BS_FP32, **EXACT)
    assert (after is None) == (alone is None), (mib, after is None)
    if after is not None:
        assert close(after, alone, 1e-6)
        worked += 1
assert worked
''',
}


@pytest.mark.parametrize("name", list(SCRIPTS))
def test_limited_pool(name):
    r = subprocess.run([sys.executable, "-c", PRELUDE % ROOT + SCRIPTS[name]], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
