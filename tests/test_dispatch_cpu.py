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


# A shard's partial sums by CTAs of 512 threads: a launch less in rounds that the host cannot enqueue as fast as they run, where few sequences
# have little work per warp (rounds of pipelined calls), or quicker in itself
@pytest.mark.parametrize("dtype,B,gamma,V,shape", [
    (F32, 1, 8, 50272, (512, 16)),   # a round 17.5 / 20.0 (from a graph 15.9 / 14.3)
    (BF16, 2, 9, 55623, (512, 16)),  # a round 17.7 / 21.5 (15.6 / 14.3)
    (F32, 7, 13, 58416, SEPARATE),   # a round 5 % less
    (F32, 10, 7, 51165, SEPARATE),   # a round 3 % less
    (F32, 19, 8, 50272, SEPARATE),   # 9.5 / 11.5 (12 CTAs)
    (BF16, 40, 16, 76000, SEPARATE),  # 22.6 / 25.0 (6 CTAs)
    (F32, 5, 6, 18928, (512, 16)),   # 3.5 / 3.9
    (F32, 38, 7, 35616, (512, 6)),   # 10.5 / 10.7
    (BF16, 48, 4, 26416, (512, 5)),  # 5.1 / 5.8
])
def test_shard_sums(L, dtype, B, gamma, V, shape):
    assert edge(L, dtype, SHARD, B, gamma, V) == shape


# Few sequences of many segments by CTAs of 512 threads, or not
@pytest.mark.parametrize("dtype,form,B,gamma,V,shape", [
    (F32, ROW, 1, 7, 50272, SEPARATE),       # 5.6 / 6.7
    (F32, ROW, 5, 2, 133456, SEPARATE),      # a round 15.3 / 15.9
    (F32, ROW, 2, 5, 48272, (512, 16)),      # a round 10.3 / 11.1
    (BF16, ROW, 33, 11, 68752, SEPARATE),    # a round 27.4 / 30.3 (6)
    (F32, FUSED, 38, 3, 24400, (512, 6)),    # 10.2 / 10.7 (256 x 10)
    (F32, BONUS, 6, 2, 109056, (512, 16)),   # a round 17.0 / 19.4
    (BF16, ROW, 12, 5, 90108, SEPARATE),     # 8.7 / 9.7
    (BF16, ROW, 19, 8, 100000, SEPARATE),    # 14.0 / 15.2
    (BF16, ROW, 30, 11, 100000, SEPARATE),   # 21.1 / 23.3
    (F32, BONUS, 1, 4, 121880, SEPARATE),    # 7.9 / 9.3
    (F32, FUSED, 44, 14, 57719, SEPARATE),   # 38.3 / 41.8
    (BF16, ROW, 2, 11, 25408, (512, 16)),    # 5.4 / 6.4
    (F32, ROW, 6, 2, 53913, (512, 16)),      # 6.5 / 7.6
    (F32, ROW, 14, 2, 83517, (512, 16)),     # 8.5 / 10.2
    (F32, ROW, 18, 11, 34312, (512, 12)),    # 10.6 / 11.4
    (F32, ROW, 29, 3, 63728, (512, 8)),      # 10.4 / 11.5
    (BF16, ROW, 45, 6, 127696, (512, 6)),    # 25.4 / 29.8
    (F32, ROW, 48, 6, 115296, (512, 5)),     # 34.4 / 35.3
    (F32, BONUS, 7, 1, 128512, (512, 16)),   # 10.0 / 13.7
    (BF16, BONUS, 27, 2, 64064, (512, 8)),   # 10.0 / 14.0
    (F32, FUSED, 17, 6, 54992, (512, 12)),   # 13.7 / 16.3
    (F32, FUSED, 1, 12, 13930, (256, 16)),   # 8.4 / 9.9 (512 threads do not hold the row)
])
def test_few_sequences(L, dtype, form, B, gamma, V, shape):
    assert edge(L, dtype, form, B, gamma, V) == shape


# CTAs of 128 threads, or not (a round where the call itself does not tell)
@pytest.mark.parametrize("dtype,form,B,gamma,V,shape", [
    (F32, ROW, 370, 12, 20480, SEPARATE),    # 76.1 / 91.2
    (F32, ROW, 220, 2, 90976, SEPARATE),     # 66.9 / 87.2 (5 CTAs)
    (BF16, ROW, 300, 4, 30011, SEPARATE),    # a round 49.5 / 49.8 (3)
    (F32, BONUS, 185, 9, 68224, SEPARATE),   # a round 122.5 / 143.4 (6)
    (BF16, FUSED, 364, 7, 23515, SEPARATE),  # 49.2 / 60.6 (3)
    (F32, FUSED, 332, 13, 1360, (256, 1)),   # 14.9 / 20.2 (3)
    (F32, FUSED, 208, 5, 6119, (256, 2)),    # 16.6 / 20.6 (5)
    (F32, ROW, 303, 2, 24064, (128, 3)),     # 22.5 / 25.6
    (F32, ROW, 359, 7, 4993, (128, 3)),      # a round 25.3 / 26.9 (256 x 1)
    (F32, ROW, 333, 10, 12288, SEPARATE),    # a round 46.0 / 54.9
    (BF16, BONUS, 350, 13, 11171, (128, 3)),  # a round 45.7 / 54.3 (256 x 1)
    (BF16, ROW, 204, 6, 5721, (512, 1)),     # a round 17.5 / 18.5 (128 x 5)
    (F32, ROW, 199, 9, 7840, (128, 5)),      # 14.9 / 15.9 (256 x 2)
    (F32, FUSED, 178, 3, 25552, (128, 6)),   # 23.7 / 27.5 (256 x 2)
    (BF16, ROW, 177, 2, 11376, (128, 6)),    # 7.0 / 8.7 (256 x 2)
])
def test_batches_of_one_or_two_ctas(L, dtype, form, B, gamma, V, shape):
    assert edge(L, dtype, form, B, gamma, V) == shape


# Pairs of CTAs as one of 512 threads, and clusters near the last that the GPU holds (a round, taken / not taken)
@pytest.mark.parametrize("dtype,form,B,gamma,V,shape", [
    (F32, ROW, 92, 14, 10400, (256, 6)),     # 20.4 / 28.7 (512 x 3)
    (BF16, ROW, 49, 9, 5242, (256, 4)),      # 10.9 / 12.2 (512 x 2)
    (BF16, ROW, 67, 7, 7744, (256, 4)),      # 9.8 / 11.2
    (F32, SHARD, 90, 7, 16752, (512, 3)),    # 26.2 / 29.5 (256 x 6)
    (BF16, ROW, 175, 4, 5280, (256, 2)),     # 11.6 / 13.2 (512 x 1)
    (F32, SHARD, 168, 7, 2048, (512, 1)),    # the call 4.0 / 4.6 (256 x 2)
    (F32, ROW, 69, 1, 95104, (512, 4)),      # 26.7 / 35.2 (256 x 8)
    (BF16, ROW, 137, 14, 44928, (512, 2)),   # 55.5 / 59.6 (256 x 4)
    (F32, ROW, 70, 2, 42528, (256, 7)),      # 22.2 / 28.8 (256 x 8)
    (F32, ROW, 75, 2, 84960, (256, 6)),      # 33.6 / 39.1 (256 x 7)
    (BF16, ROW, 108, 3, 61178, (256, 4)),    # 36.0 / 40.2 (256 x 5)
])
def test_pairs_and_full_waves(L, dtype, form, B, gamma, V, shape):
    assert edge(L, dtype, form, B, gamma, V) == shape


# The edge's draw of bonus tokens in the same launch, or not
@pytest.mark.parametrize("dtype,B,gamma,V,shape", [
    (F32, 1, 5, 57440, SEPARATE),     # 7.5 / 11.4 (256 x 8)
    (F32, 1, 8, 42042, SEPARATE),     # 7.6 / 11.2
    (F32, 3, 5, 58288, (512, 16)),    # a round 12.3 / 15.4
    (BF16, 2, 10, 31702, (256, 8)),   # 9.3 / 10.4 (the row is held)
])
def test_bonus_draws(L, dtype, B, gamma, V, shape):
    assert edge(L, dtype, BONUS, B, gamma, V) == shape


def draw(L, B, V):
    t, c, turns = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    L.dssd_test_draw_shape(B, V, ctypes.byref(t), ctypes.byref(c), ctypes.byref(turns))
    return t.value, c.value, turns.value


# Draws in turns by one CTA per sequence: all CTAs resident, forty warps of an SM in whole CTAs
@pytest.mark.parametrize("B,V,shape", [
    (740, 20480, (256, 1, 1)),    # 17.2 / 19.0 (two kernels)
    (741, 12800, (192, 1, 1)),    # five CTAs of seven warps are 740
    (914, 14080, (0, 0, 0)),      # 18.2 / 20.9 (192 x 1: six CTAs of six warps are 888)
    (795, 16068, (0, 0, 0)),      # 15.0 / 17.2 (224 x 1)
    (915, 12480, (160, 1, 1)),    # (192 x 1 20.8, two kernels 18.2)
    (1000, 12288, (160, 1, 1)),   # 15.6 / 17.4
    (1400, 10240, (128, 1, 1)),   # 16.8 / 20.5
    (1480, 4612, (128, 1, 1)),    # ten CTAs of four warps are 1480
    (1481, 4612, (0, 0, 0)),
])
def test_draws_by_one_cta(L, B, V, shape):
    assert draw(L, B, V) == shape


# Draws in turns by clusters, by one CTA while the wave is not full, and of few long rows
@pytest.mark.parametrize("B,V,shape", [
    (383, 23016, (0, 0, 0)),      # 13.5 / 15.2 (128 x 3)
    (406, 18672, (0, 0, 0)),      # 12.2 / 14.2 (128 x 3)
    (330, 23040, (128, 3, 1)),    # 11.9 / 13.1
    (290, 19376, (128, 3, 1)),    # 9.6 / 10.6 (128 x 4; two kernels 9.6)
    (340, 15924, (256, 1, 1)),    # a round 24.7 / 26.7 (128 x 3)
    (105, 17084, (128, 5, 1)),    # a round 15.2 / 17.4 (256 x 5)
    (352, 19047, (0, 0, 0)),      # 13.6 / 17.3 (256 x 1)
    (400, 18218, (0, 0, 0)),      # 14.3 / 16.2
    (92, 20030, (0, 0, 0)),       # 7.1 / 8.3 (128 x 5)
    (133, 15897, (0, 0, 0)),      # 7.4 / 8.8 (128 x 4)
    (105, 17034, (0, 0, 0)),      # 7.5 / 9.0 (256 x 5)
    (107, 22920, (0, 0, 0)),      # 6.4 / 7.2 (128 x 6)
    (141, 17020, (128, 5, 1)),    # 7.0 / 9.6 (two kernels)
    (251, 4608, (128, 3, 1)),     # 5.7 / 6.4 (256 x 1)
    (290, 5120, (128, 3, 1)),     # 5.9 / 6.3 (256 x 1)
    (318, 4880, (256, 1, 1)),     # 6.9 / 8.3 (128 x 3)
    (340, 4608, (256, 1, 1)),     # 6.5 / 8.0
])
def test_draws_in_turns(L, B, V, shape):
    assert draw(L, B, V) == shape
