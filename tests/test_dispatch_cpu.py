"""Which kernels a size takes, at sizes that were timed with both: the quicker ones (microseconds a call, taken / not taken)."""
import ctypes

import pytest

ROW, BONUS, FUSED, SHARD = range(4)
F32, BF16 = 0, 1
SEPARATE = (0, 0)


@pytest.fixture(scope="module")
def L():
    from paper_2507_12000_b200 import build

    build.build()
    from paper_2507_12000_b200 import binding

    return binding.lib


def edge(L, dtype, form, B, gamma, V):
    t, c = ctypes.c_int(), ctypes.c_int()
    L.dssd_test_edge_shape(dtype, form, B, gamma, V, ctypes.byref(t), ctypes.byref(c))
    return t.value, c.value


# A shard's partial sums by CTAs of 512 threads: about a segment per warp in clusters of more than eight CTAs, up to three in smaller ones
@pytest.mark.parametrize("dtype,B,gamma,V,shape", [
    (F32, 1, 8, 50272, SEPARATE),    # 3.7 / 5.2 (16 CTAs)
    (F32, 4, 5, 50272, SEPARATE),    # 4.0 / 5.0
    (BF16, 8, 4, 76000, SEPARATE),   # 4.4 / 5.0
    (F32, 14, 4, 60000, SEPARATE),   # 5.2 / 6.3
    (F32, 19, 8, 50272, SEPARATE),   # 9.5 / 11.5 (12 CTAs)
    (BF16, 40, 16, 76000, SEPARATE),  # 22.6 / 25.0 (6 CTAs)
    (F32, 5, 6, 18928, (512, 16)),   # 3.5 / 3.9
    (F32, 38, 7, 35616, (512, 6)),   # 10.5 / 10.7
    (BF16, 48, 4, 26416, (512, 5)),  # 5.1 / 5.8
])
def test_shard_sums(L, dtype, B, gamma, V, shape):
    assert edge(L, dtype, SHARD, B, gamma, V) == shape
