"""The truncated-support round where its geometry can go wrong: vocabularies at the edges of a tile of the
selection kernel (4096 float32 or 8192 bf16 logits), launches at the thresholds of one / two / four tiles per
CTA, the smallest and the largest k, rows whose runs hold fewer than k entries, rows that are masked (mostly
-inf), and runs whose candidates overflow the buffer."""
import numpy as np
import pytest

import dssd_inputs as di
from test_parity_topk_gpu import compare_topk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_12000_b200 import binding

    return binding


@pytest.mark.parametrize("dtype,Bn,gamma,V,k", [
    ("f32", 3, 1, 4095, 32), ("f32", 3, 1, 4096, 1), ("f32", 3, 1, 4099, 10), ("bf16", 3, 2, 8191, 32), ("bf16", 3, 2, 8192, 10),
    ("bf16", 3, 2, 8200, 32), ("bf16", 2, 1, 16400, 32), ("f32", 4, 15, 9000, 10), ("f32", 4, 16, 9001, 10),
    ("f32", 587, 1, 16384, 10), ("f32", 588, 1, 16384, 10), ("f32", 791, 2, 32768, 4), ("f32", 792, 2, 32768, 32),
    ("f32", 2, 1, 600001, 32), ("bf16", 3, 2, 8200, 12), ("bf16", 3, 2, 8200, 13), ("f32", 3, 2, 200, 20), ("bf16", 800, 2, 65536, 32),
])
def test_round_at_the_edges(B, oracle_mod, dtype, Bn, gamma, V, k):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.5, seed=V + Bn)
    compare_topk(B, oracle_mod, di.generate_topk(w, k, threads=16), w.temperature, k)


@pytest.mark.parametrize("k", [1, 10, 32])
def test_masked_and_overflowing_rows(B, oracle_mod, k):
    """Rows that keep a few entries above -inf (fewer and more than k), runs that repeat one value, and a first
    tile of equal logits followed by larger ones."""
    Bn, gamma, V = 5, 2, 30000
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype="f32", temperature=0.9, sigma_d=0.5, seed=k)
    d = di.generate_topk(w, k, threads=4)
    tl = d["target_logits"]
    rng = np.random.default_rng(k)
    for b, keep in ((0, 5), (1, 40)):
        mask = np.ones(V, bool)
        mask[rng.choice(V, keep, replace=False)] = False
        tl[b][:, mask] = -np.inf
    tl[2] = np.repeat(np.arange(V // 100, dtype=np.float32), 100)[None]
    tl[3][:, :4096] = 0.0
    tl[3][:, 4096:] = np.linspace(0.0, 1.0, V - 4096, dtype=np.float32)[None]
    compare_topk(B, oracle_mod, d, w.temperature, k)


@pytest.mark.parametrize("k", [1, 9, 10, 32])
@pytest.mark.parametrize("dtype,Bn,gamma,V", [("f32", 9, 1, 30011), ("bf16", 9, 1, 30011), ("bf16", 520, 2, 32768), ("f32", 520, 4, 33003)])
def test_ties_and_masks(B, oracle_mod, dtype, Bn, gamma, V, k):
    """Runs whose candidates overflow: masks of several values (ties at the threshold, of which the lowest indices count) that end
    anywhere, ascending rows, few distinct values, and rows with more candidates above any bound from the threads'
    maxima than fit; in rows at every alignment, in runs of one, two and four tiles."""
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype="f32", temperature=0.9, sigma_d=0.5, seed=k)
    d = di.generate_topk(w, k, threads=16)
    tl = d["target_logits"]
    rng = np.random.default_rng(k)
    at = np.arange(V)
    for i, low in ((0, -1.0e9), (1, -10000.3), (2, np.finfo(np.float32).min), (3, -np.inf)):
        tl[i][:, rng.random(V) < 0.9995 if i % 2 else at >= 17] = low
    tl[4][:] = np.linspace(-1.0, 1.0, V, dtype=np.float32)
    tl[5][:] = 0.1234567
    tl[6][:] = rng.integers(0, 3, V)
    tl[7][:] = np.where(at // 4 % 128 < 32, 0.0, 1.0 + at / V)
    tl[8][:, : V // 2], tl[8][:, V // 2:] = -0.0, 0.0
    if dtype == "bf16":
        with np.errstate(over="ignore"):
            d["target_logits"] = (np.where(np.abs(tl) == np.finfo(np.float32).max, np.sign(tl) * 3.3e38, tl).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    compare_topk(B, oracle_mod, d, w.temperature, k)


@pytest.mark.parametrize("V,k", [(4 * 4096, 20), (5 * 4096, 20), (3 * 4096, 32), (9 * 4096, 29), (33 * 4096 + 5, 8), (30 * 4096, 32), (33 * 4096, 32), (300 * 4096 + 1, 1), (300 * 4096, 10),
                                 (300 * 4096 + 3, 32), (2100 * 4096, 12)])
def test_rows_of_many_runs(B, oracle_mod, V, k):
    """Merging the lists of many runs (4096 float32 entries each), all keys and only those of the lists that matter: equal shares, rows
    whose best entries lie in fewer of the merging lanes than the bound needs (so that hundreds of keys and lists reach it), ascending
    rows, and rows with fewer than k entries above -inf."""
    w = di.custom(B=4, gamma=0 if V > 5000000 else 1, V=V, dtype="f32", temperature=0.9, sigma_d=0.5, seed=k)
    d = di.generate_topk(w, k, threads=16)
    tl, run = d["target_logits"], np.arange(V) // 4096
    tl[1] += np.where(run % 32 < 15, 50.0, 0.0).astype(np.float32)
    tl[2][:] = np.linspace(-3.0, 9.0, V, dtype=np.float32)
    tl[3][:, np.arange(V) % 9001 != 0] = -np.inf
    compare_topk(B, oracle_mod, d, w.temperature, k)


@pytest.mark.parametrize("Bn,gamma,V,k", [(3, 31, 9000, 10), (3, 32, 9000, 10), (2, 63, 20000, 32), (9, 64, 300, 5), (2, 200, 70000, 12),
                                          (1, 1000, 64, 13)])
def test_many_positions(B, oracle_mod, Bn, gamma, V, k):
    """Positions in turns and, beyond two turns, judged by a kernel of their own: rejections at any position, rows without a
    distribution before and after them, draft tokens out of range."""
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype="f32", temperature=0.9, sigma_d=0.2, seed=k)
    d = di.generate_topk(w, k, threads=16)
    d["uniforms"][0] = 0.0  # accepted wherever the token is in the support
    for i in range(1, Bn):
        d["uniforms"][i, : gamma * i // Bn] = 0.0
        d["uniforms"][i, gamma * i // Bn] = 1.0
    d["target_logits"][0, gamma // 2, 7] = np.nan
    d["draft_tokens"][-1, -1] = V
    compare_topk(B, oracle_mod, d, w.temperature, k)


@pytest.mark.parametrize("k", [4, 8, 9, 10, 17, 31, 32])
def test_draw_sums_in_index_order(B, oracle_mod, k):
    """The draw's sums are those of a loop over the entries in index order, bit for bit, bonus and residual: entries so much smaller than
    the sum before them that sums in another order end elsewhere, and uniforms on the steps of the distribution."""
    import torch

    Bn, gamma = 512, 1
    rng = np.random.default_rng(k)
    p = np.ldexp(rng.uniform(0.5, 1.0, (Bn, k)), -rng.integers(0, 64, (Bn, k))).astype(np.float32)
    p[0], p[1] = 2.0 ** -55, 2.0 ** -54
    p[:2, 0] = p[:2, k - 1] = 0.5  # (sum 1; the entries between weigh nothing one by one)
    idx = np.sort(np.stack([rng.choice(100000, k, replace=False) for _ in range(Bn)]), axis=1).astype(np.int32)
    n = (np.arange(Bn) % 3 != 2).astype(np.int32) * gamma  # a third of them residual draws, from q = 0 but for one entry
    q_idx, q_val = np.full((Bn, gamma, k), 200000, np.int32), np.zeros((Bn, gamma, k), np.float32)
    q_idx[:, 0, 0], q_val[:, 0, 0] = idx[:, k // 2], 0.25 * p[:, k // 2]
    r = np.where((n[:, None] < gamma) & (np.arange(k) == k // 2), 0.75, 1.0) * p.astype(np.float64)
    C = np.zeros((Bn, k))
    s = np.zeros(Bn)
    for e in range(k):
        s = s + r[:, e]
        C[:, e] = s
    u = np.minimum(C[np.arange(Bn), rng.integers(0, k, Bn)] / s, 1 - 2.0 ** -24).astype(np.float32)
    u[:2] = 0.5
    over = C > (u.astype(np.float64) * s)[:, None]
    want = np.where(over.any(axis=1), idx[np.arange(Bn), over.argmax(axis=1)], idx[:, k - 1])
    ref = oracle_mod.device_resample_topk(idx, p, q_idx, q_val, n, u, gamma)
    assert (ref["token"] == want).all()
    up = lambda a: torch.from_numpy(a).cuda()
    got = B.dssd_device_resample_topk(up(idx), up(p), up(q_idx), up(q_val), up(n), up(u), gamma)
    torch.cuda.synchronize()
    assert (got["token"].cpu().numpy() == want).all()
