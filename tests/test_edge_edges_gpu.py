"""The edge half where its geometry can go wrong: vocabularies at the edges of a tile of the log-sum-exp
kernel (4096 float32 or 8192 bf16 logits), of a segment of the one-launch kernel and of the emission (8192 entries), launches
at the thresholds of one / two / four tiles per CTA and of folding inside the emission, 32 positions and more per
sequence.  (Sequences of 33 positions and more always take the separate kernels.)"""
import pytest

import dssd_inputs as di
from gpu_util import compare_round
from test_parity_bonus_gpu import compare_bonus
from test_parity_dsd_gpu import compare_dsd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_12000_b200 import binding

    return binding


@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 2, 2, 1), ("bf16", 2, 2, 7), ("f32", 3, 1, 4095), ("f32", 3, 1, 4096), ("f32", 3, 1, 4099),
    ("bf16", 3, 2, 8191), ("bf16", 3, 2, 8192), ("bf16", 3, 2, 8193), ("f32", 2, 1, 8200), ("bf16", 2, 0, 16385),
    ("f32", 4, 31, 3000), ("bf16", 4, 32, 3001), ("f32", 2, 64, 1500),
    ("bf16", 592, 1, 600), ("bf16", 593, 1, 600), ("f32", 74, 1, 65536), ("f32", 75, 1, 65536),
    ("f32", 587, 1, 16384), ("f32", 588, 1, 16384), ("f32", 791, 2, 32768), ("f32", 792, 2, 32768),
    ("bf16", 1600, 2, 36001), ("bf16", 5, 1, 8189), ("bf16", 5, 1, 8190), ("f32", 5, 1, 8191), ("f32", 5, 2, 16385),
])
def test_round_at_the_edges(B, oracle_mod, dtype, Bn, gamma, V):
    """Whichever kernels the sizes take."""
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.5, zipf=V > 8, seed=V + Bn)
    compare_round(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


# The separate kernels: rows shorter than a vector, a tile and its neighbours, one, two and four tiles per CTA (2970 and 3003, 18975 and
# 19008 tiles in all), folds in the emission and in a kernel of their own (592 and 593 emission CTAs).
@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 2, 32, 1), ("bf16", 2, 32, 7), ("f32", 3, 32, 4095), ("f32", 3, 32, 4096), ("f32", 3, 32, 4099), ("bf16", 3, 33, 8191),
    ("bf16", 3, 33, 8192), ("bf16", 3, 33, 8193), ("bf16", 2, 32, 8200), ("f32", 2, 40, 16385), ("f32", 90, 32, 4096), ("f32", 91, 32, 4096),
    ("f32", 575, 32, 4096), ("f32", 576, 32, 4096), ("bf16", 592, 32, 600), ("bf16", 593, 32, 600), ("f32", 40, 8, 70001), ("f32", 300, 4, 16384),
])
def test_separate_kernels_at_the_edges(B, oracle_mod, dtype, Bn, gamma, V):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.3, zipf=V > 8, seed=V + Bn)
    compare_round(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


# Rows of more runs than eight threads add up in two looks (64 of 4096 float32 or 8192 bf16 logits): a warp per row in the fold, more
# rows than warps, more than 32 positions.
@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 1, 2, 262144), ("f32", 1, 2, 262148), ("f32", 2, 40, 300001), ("bf16", 3, 9, 540001), ("f32", 1, 1, 1100003), ("bf16", 1, 1, 5000001),
])
def test_rows_of_many_runs(B, oracle_mod, dtype, Bn, gamma, V):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.3, zipf=True, seed=V + Bn)
    compare_round(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


# One launch for small sequences: vocabularies at the edges of a warp's segment (1024 float32 or 2048 bf16 logits) and
# of what it emits (512 entries), one CTA per sequence, clusters of two, eight, nine and sixteen, the last
# batch of a wave, the most positions, and the sizes next to the limits where the separate kernels take over.
@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 1, 1, 1023), ("f32", 1, 3, 1024), ("f32", 3, 3, 1025), ("f32", 3, 15, 1027), ("bf16", 2, 3, 2047), ("bf16", 2, 3, 2048),
    ("bf16", 2, 7, 2049), ("bf16", 3, 3, 2055), ("bf16", 1, 7, 16384), ("bf16", 1, 8, 16384), ("f32", 36, 15, 8192), ("f32", 37, 15, 8195),
    ("f32", 38, 15, 8192), ("f32", 73, 7, 8192), ("bf16", 74, 7, 16389), ("bf16", 296, 5, 5000), ("bf16", 297, 5, 5000), ("f32", 593, 3, 2500),
    ("f32", 30, 30, 2000), ("f32", 3, 31, 2100), ("bf16", 3, 32, 2100), ("f32", 185, 31, 12289), ("bf16", 8, 5, 81776), ("bf16", 4, 2, 58880),
])
def test_one_launch_at_the_edges(B, oracle_mod, dtype, Bn, gamma, V):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.5, zipf=True, seed=V + Bn)
    compare_round(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


# The same launch with the draw in it (bonus at the edge; fused verification): rows held by the cluster's warps, with 16
# CTAs and with one, and streamed, at the batch where the one ends and the other begins; segments of 512 entries at their
# edges; residuals without mass, which fall back to the row itself.
@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 1, 2, 511), ("f32", 2, 2, 512), ("bf16", 3, 3, 513), ("bf16", 2, 1, 4096), ("bf16", 2, 1, 4097), ("f32", 3, 5, 16383),
    ("bf16", 8, 4, 32000), ("f32", 4, 7, 20006), ("f32", 100, 3, 2048), ("f32", 101, 3, 2048), ("bf16", 200, 2, 1500), ("bf16", 201, 2, 1501),
    ("f32", 64, 4, 9001), ("bf16", 592, 3, 3001), ("bf16", 600, 3, 6000), ("f32", 66, 15, 6240), ("f32", 130, 3, 33000),
])
def test_draws_in_the_same_launch(B, oracle_mod, dtype, Bn, gamma, V):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.4, zipf=True, seed=V + Bn)
    d = di.generate(w, threads=16)
    compare_bonus(B, oracle_mod, d, w.temperature, threads=16)
    d["draft_q"][: (Bn + 1) // 2] = 1.0  # rejected nearly always, and max(0, p - q) is 0 everywhere
    d["draft_q_tok"][: (Bn + 1) // 2] = 1.0
    compare_dsd(B, oracle_mod, d, w.temperature, threads=16)


# Other CTAs than those of 256 threads: of 512 for sequences of many segments (at the batches where their number per sequence
# changes) and for pairs in full launches, of 128 for batches that would leave a sequence one CTA; and launches that
# spread over twice the CTAs; with and without a draw.
@pytest.mark.parametrize("dtype,Bn,gamma,V", [
    ("f32", 14, 6, 37623), ("bf16", 15, 8, 52000), ("f32", 19, 7, 20000), ("f32", 20, 7, 20001), ("f32", 30, 7, 17000), ("f32", 31, 7, 17003),
    ("bf16", 45, 7, 40000), ("bf16", 46, 7, 40000), ("f32", 52, 8, 13000), ("f32", 53, 8, 13000), ("bf16", 1, 3, 80000),
    ("bf16", 300, 4, 9792), ("f32", 332, 13, 5816), ("f32", 203, 10, 7681), ("bf16", 185, 7, 8193), ("f32", 371, 5, 4100),
    ("bf16", 117, 2, 6656), ("bf16", 61, 11, 7500), ("f32", 259, 3, 14848), ("bf16", 3, 15, 4160), ("f32", 23, 7, 2286), ("bf16", 35, 1, 8200),
])
def test_other_cta_sizes(B, oracle_mod, dtype, Bn, gamma, V):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.4, zipf=True, seed=V + Bn)
    d = di.generate(w, threads=16)
    compare_round(B, oracle_mod, d, w.temperature, threads=16)
    compare_bonus(B, oracle_mod, d, w.temperature, threads=16)
    compare_dsd(B, oracle_mod, d, w.temperature, threads=16)


def _shape(B, dtype, form, Bn, gamma, V):
    import ctypes

    t, c = ctypes.c_int(), ctypes.c_int()
    B.lib.dssd_test_edge_shape(int(dtype == "bf16"), form, Bn, gamma, V, ctypes.byref(t), ctypes.byref(c))
    return t.value, c.value


# The last batch of each row of the tables of other CTA sizes and the first beyond it, and as many partial sums as a CTA's shared
# memory holds (1024: sixteen positions of 64 segments, eight of 128) and one segment more per row.
@pytest.mark.parametrize("dtype,Bn,gamma,V,shape", [
    ("f32", 8, 2, 53913, (512, 16)), ("f32", 9, 2, 53913, (512, 16)), ("f32", 14, 2, 83517, (512, 16)), ("f32", 15, 2, 53913, (512, 12)),
    ("f32", 19, 11, 17000, (512, 12)), ("f32", 20, 3, 63728, (512, 8)), ("f32", 30, 3, 63728, (512, 8)), ("f32", 31, 9, 26000, (512, 6)),
    ("f32", 45, 7, 20000, (512, 6)), ("f32", 46, 7, 20000, (512, 5)), ("f32", 52, 7, 20000, (512, 5)), ("f32", 53, 7, 20000, (256, 8)),
    ("f32", 181, 4, 4200, (128, 6)), ("f32", 182, 4, 4200, (128, 5)), ("f32", 204, 4, 4200, (128, 5)), ("f32", 205, 4, 4200, (512, 1)),
    ("f32", 370, 4, 4200, (128, 3)), ("f32", 371, 4, 4200, (256, 1)), ("bf16", 177, 2, 11376, (128, 6)), ("f32", 65, 7, 8200, (256, 8)), ("f32", 66, 7, 8200, (512, 4)),
    ("f32", 45, 15, 65536, (512, 6)), ("f32", 45, 15, 65540, (0, 0)),
])
def test_edges_of_the_tables(B, oracle_mod, dtype, Bn, gamma, V, shape):
    assert _shape(B, dtype, 0, Bn, gamma, V) == shape
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.4, zipf=True, seed=V + Bn)
    compare_round(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


@pytest.mark.parametrize("V,shape", [(131072, (512, 16)), (131076, (0, 0))])
def test_as_many_partial_sums_as_fit_with_a_draw(B, oracle_mod, V, shape):
    assert _shape(B, "f32", 1, 14, 7, V) == shape
    w = di.custom(B=14, gamma=7, V=V, dtype="f32", temperature=0.9, sigma_d=0.1, zipf=True, seed=V)
    compare_bonus(B, oracle_mod, di.generate(w, threads=16), w.temperature, threads=16)


# Residuals without mass, drawn for by CTAs of 128 and of 512 threads
@pytest.mark.parametrize("dtype,Bn,gamma,V,shape", [
    ("f32", 178, 3, 9000, (128, 6)), ("bf16", 187, 4, 12384, (128, 5)), ("f32", 320, 3, 8193, (128, 3)), ("f32", 17, 6, 54992, (512, 12)), ("bf16", 2, 3, 75001, (512, 16)),
])
def test_fallback_of_other_cta_sizes(B, oracle_mod, dtype, Bn, gamma, V, shape):
    assert _shape(B, dtype, 2, Bn, gamma, V) == shape
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.4, zipf=True, seed=V + Bn)
    d = di.generate(w, threads=16)
    d["draft_q"][: (Bn + 1) // 2] = 1.0  # rejected nearly always, and max(0, p - q) is 0 everywhere
    d["draft_q_tok"][: (Bn + 1) // 2] = 1.0
    compare_dsd(B, oracle_mod, d, w.temperature, threads=16)


@pytest.mark.parametrize("dtype,V,stride", [("bf16", 4096, 1), ("bf16", 40000, 97), ("f32", 4096, 1)])
def test_every_entry_of_a_vector_counts(B, dtype, V, stride):
    """Some terms of a row's sum are formed by a polynomial, the others by the special-function unit: a NaN is seen in
    every position, -inf and terms far below the largest weigh nothing, and a row of one entry above -inf is 1 there."""
    import torch

    Bn, dt = 40, torch.bfloat16 if dtype == "bf16" else torch.float32
    at = torch.arange(Bn, device="cuda") * stride
    rows = torch.arange(Bn, device="cuda")
    none = torch.empty(Bn, 0, device="cuda")
    run = lambda z: B.dssd_edge_verify(z.view(Bn, 1, V), none.int(), none, none, 1.0)
    z = torch.zeros(Bn, V, dtype=dt, device="cuda")
    z[rows, at] = float("nan")
    assert (run(z)["flags"] == B.EDGE_FLAG_NONFINITE).all()
    for low in (float("-inf"), -1.0e4, -200.0, -90.0):
        z = torch.full((Bn, V), low, dtype=dt, device="cuda")
        z[rows, at] = 1.5
        ev = run(z)
        assert (ev["flags"] == 0).all()
        assert ((ev["p_row"][rows, at] - 1.0).abs() <= 3e-7).all() and ((ev["lse"][:, 0] - 1.5).abs() <= 1e-6).all()
    z = torch.zeros(Bn, V, dtype=dt, device="cuda")  # equal entries: n in all positions
    assert ((run(z)["p_row"] * V - 1.0).abs() <= 2e-6).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("Bn,gamma,V", [(1, 0, 40000), (8, 4, 32000), (300, 4, 30011), (40, 8, 70001), (256, 4, 151936)])
def test_masks_of_the_lowest_value_weigh_nothing(B, dtype, Bn, gamma, V):
    """Masks of the type's lowest value, whose scaled logits are below float32's range, give bit for bit what masks of -inf
    give, wherever they begin and end: whole tiles of a thread, its first ones, all but one entry."""
    import torch

    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    z = torch.randn(Bn, gamma + 1, V, device="cuda", generator=torch.Generator("cuda").manual_seed(V)).to(dt)
    x = torch.zeros(Bn, gamma, dtype=torch.int32, device="cuda")
    half = torch.full((Bn, gamma), 0.5, device="cuda")
    for a, b in ((0, V // 2), (0, 24576), (8192, V), (16384, 32768), (V // 3, V), (1, V), (0, V - 1)):
        got = []
        for low in (torch.finfo(dt).min, float("-inf")):
            masked = z.clone()
            masked[:, :, a:b] = low
            got.append(B.dssd_edge_verify(masked, x, half, half, 1.0))
        assert (got[0]["flags"] == 0).all()
        for k in ("accept_len", "p_row", "lse", "flags", "p_tok"):
            assert torch.equal(got[0][k], got[1][k]), (k, a, b)
    rows = torch.full((Bn, gamma + 1, V), torch.finfo(dt).min, dtype=dt, device="cuda")  # nothing inside the range
    assert (B.dssd_edge_verify(rows, x, half, half, 1.0)["flags"] == B.EDGE_FLAG_NONFINITE).all()
