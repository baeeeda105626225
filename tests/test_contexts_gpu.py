"""The library in a process with several contexts on one device, one after the other and in turn: what it keeps per context
(the permission for clusters of more than eight CTAs) is asked for in each.  Runs in a process of its own, through the C ABI."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
c = ctypes
cu, L = c.CDLL("libcuda.so.1"), c.CDLL(sys.argv[1])
L.dssd_edge_verify.argtypes = [c.c_void_p, c.c_int, c.c_int64, c.c_void_p, c.c_void_p, c.c_void_p, c.c_float, c.c_int, c.c_int, c.c_int,
                               c.c_void_p, c.c_void_p, c.c_void_p, c.c_void_p, c.c_void_p, c.c_void_p, c.c_size_t, c.c_void_p]
L.dssd_edge_verify_workspace_bytes.restype = c.c_size_t
gamma, V = 8, 16384  # 72 segments of a warp: nine CTAs in a cluster

def ok(st):
    assert st == 0, st

def alloc(n, word=0):
    p = c.c_uint64()
    ok(cu.cuMemAlloc_v2(c.byref(p), c.c_size_t(n)))
    ok(cu.cuMemsetD32_v2(p, c.c_uint(word), c.c_size_t(n // 4)))
    return p.value

def round_():
    n = alloc(4, 77)
    nb = L.dssd_edge_verify_workspace_bytes(1, gamma, V)
    st = L.dssd_edge_verify(alloc((gamma + 1) * V * 2), 1, V, alloc(4 * gamma), alloc(4 * gamma, 0x38000000), alloc(4 * gamma, 0x3f000000), 1.0,
                            1, gamma, V, n, alloc(4 * V), None, None, None, alloc(nb), nb, None)
    assert st == 0, (st, L.dssd_last_cuda_error())
    ok(cu.cuCtxSynchronize())
    got = c.c_int()
    ok(cu.cuMemcpyDtoH_v2(c.byref(got), c.c_uint64(n), c.c_size_t(4)))
    assert got.value == gamma, got.value  # p = 1 / V = 2 q: everything is accepted

ok(cu.cuInit(0))
first, second, third = c.c_void_p(), c.c_void_p(), c.c_void_p()
ok(cu.cuCtxCreate_v2(c.byref(first), 0, 0))
round_()
ok(cu.cuCtxCreate_v2(c.byref(second), 0, 0))
round_()
ok(cu.cuCtxSetCurrent(first))
round_()
ok(cu.cuCtxDestroy_v2(first))
ok(cu.cuCtxSetCurrent(second))
round_()
ok(cu.cuCtxDestroy_v2(second))
ok(cu.cuCtxCreate_v2(c.byref(third), 0, 0))
round_()
print("fine")
"""


def test_one_context_after_the_other():
    from paper_2507_12000_b200 import binding

    r = subprocess.run([sys.executable, "-c", CHILD, binding.LIB_PATH], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "fine", (r.stdout[-500:], r.stderr[-2000:])
