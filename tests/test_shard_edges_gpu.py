"""The vocabulary-sharded round where its geometry can go wrong: more shards than are requested at once (8) and
than a warp has lanes, slices at the edges of what a cluster of CTAs holds, batches at its threshold."""
import pytest

import dssd_inputs as di
from test_parity_shard_gpu import B, compare_sharded  # noqa: F401  (B is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,V,gamma,Bn,G", [
    ("f32", 9000, 2, 4, 9), ("bf16", 20000, 1, 3, 33), ("f32", 40, 2, 3, 40), ("f32", 65536, 2, 25, 2), ("f32", 65536, 1, 26, 2),
    ("bf16", 65538, 1, 5, 2), ("f32", 131072, 1, 3, 2), ("f32", 131080, 1, 3, 2), ("bf16", 2000, 2, 200, 2), ("bf16", 2000, 2, 201, 2),
    ("f32", 2046, 3, 3, 2), ("bf16", 4097, 3, 3, 2), ("bf16", 4100, 31, 3, 2), ("bf16", 4100, 32, 3, 2), ("f32", 16384, 7, 2, 2), ("bf16", 16390, 2, 592, 2), ("f32", 33000, 8, 30, 2),
    ("f32", 75246, 6, 3, 2), ("bf16", 19584, 4, 300, 2), ("f32", 4096, 7, 168, 2), ("bf16", 13000, 7, 13, 2),
    ("f32", 1048576, 1, 2, 2),
    # CTAs of 128 threads, which add up sixteen positions at a time
    ("bf16", 8622, 14, 200, 2), ("bf16", 8622, 15, 200, 2), ("bf16", 8622, 16, 200, 2), ("f32", 6000, 31, 200, 2),
    ("bf16", 1048602, 1, 2, 2), ("f32", 1200007, 1, 2, 1),
])
def test_round_at_the_edges(B, dtype, V, gamma, Bn, G):  # noqa: F811
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.8, sigma_d=0.8, seed=V + G)
    compare_sharded(B, di.generate(w, threads=8), w.temperature, G)
