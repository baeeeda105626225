"""The dense draw where its geometry can go wrong: vocabularies at the edges of a chunk (1024 entries) and of
a tile (4096), batches at the thresholds of tiles per CTA, more chunks than a warp's lanes keep in
registers, one sum per tile instead of per chunk, aligned and unaligned rows, both payloads; uniforms at
both ends of their range and rows whose mass sits in single entries."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_12000_b200 import binding

    return binding


@pytest.mark.parametrize("Bn,gamma,V,half", [
    (5, 2, 1, False), (5, 2, 1023, False), (5, 2, 1024, True), (5, 1, 1025, False), (5, 3, 4095, True),
    (5, 2, 4096, False), (5, 2, 4097, False), (7, 1, 4100, True), (3, 1, 8192, False), (3, 1, 12289, False),
    (9, 2, 511, False), (9, 2, 513, True), (25, 1, 32768, False), (26, 1, 32768, False), (3, 2, 32769, False), (6, 1, 65536, True),
    (7, 1, 65536, False), (4, 2, 65537, False), (200, 1, 900, False), (201, 1, 900, True), (5, 1, 50257, True), (1199, 1, 4096, False), (1200, 1, 4096, False), (150, 1, 32768, True), (4801, 1, 4000, False),
    (600, 1, 4096, False), (601, 1, 4096, True), (1200, 1, 2047, True), (1201, 1, 2047, False), (2400, 1, 1024, False), (2401, 1, 1024, False),
    (6, 2, 9001, False), (6, 3, 9002, True), (7, 2, 9003, True), (6, 2, 9003, False), (600, 1, 36864, False), (2, 1, 262144, False), (2, 1, 266241, False), (1200, 1, 114700, True), (32768, 1, 4097, False), (32769, 1, 8193, True),
    # clusters of 128, 256 and 512 threads that hold a row: at and beyond eight and sixteen CTAs and the waves they are chosen for
    (40, 1, 16384, False), (40, 1, 16385, True), (45, 1, 16896, False), (46, 1, 16896, True), (187, 2, 6144, False), (188, 2, 6144, False),
    (12, 1, 65536, False), (13, 1, 65533, False), (4, 1, 131072, True), (4, 1, 131073, False), (5, 2, 131072, False),
    # rows in turns: as many warps as segments, one CTA per sequence in one to five turns, clusters, and beyond
    (100, 1, 18432, False), (101, 1, 18432, True), (330, 2, 4500, False), (719, 1, 12001, False), (740, 1, 20480, False), (740, 1, 20481, True),
    (1180, 1, 9001, True), (1201, 1, 2044, False), (150, 2, 23040, False), (150, 2, 23041, False),
    (740, 1, 12800, False), (741, 1, 12800, False), (888, 1, 9000, False), (889, 1, 9000, True), (914, 1, 14080, False), (915, 1, 12480, False), (149, 1, 20992, False), (149, 1, 20993, True),
    (350, 1, 11248, False), (351, 1, 11248, False), (319, 1, 6144, False), (320, 1, 6144, True), (290, 1, 19376, False),
    (3, 1, 1 << 19, False), (3, 1, (1 << 19) + 1, False), (4, 1, 1 << 20, False), (4, 1, (1 << 20) + 1, True), (3, 1, (1 << 21) + 3, False), (3, 1, 5000001, False),
])
def test_draw_at_the_edges(B, oracle_mod, Bn, gamma, V, half):
    gen = torch.Generator(device="cuda").manual_seed(Bn + V)
    p = torch.softmax(2.0 * torch.randn(Bn, V, generator=gen, device="cuda"), dim=-1)
    q = torch.softmax(2.0 * torch.randn(Bn, gamma, V, generator=gen, device="cuda"), dim=-1)
    if V > 1:
        p[0] = 0.0
        p[0, V - 1] = 1.0          # all mass in the last entry
        p[1] = 0.0
        p[1, V // 2] = 0.5         # two entries, the draw falls on the second with u = 1/2
        p[1, V - 1] = 0.5
    n = (torch.arange(Bn, device="cuda") % (gamma + 1)).to(torch.int32)
    n[1] = gamma                   # bonus draws, where r = p
    u = torch.randint(0, 1 << 24, (Bn,), generator=gen, device="cuda").to(torch.float32) * 2.0 ** -24
    u[1] = 0.5
    u[2 % Bn] = 0.0
    u[-1] = 1.0 - 2.0 ** -24
    if half:
        p = p.to(torch.float16)
    out = B.dssd_device_resample(p, q, n, u, gamma)
    torch.cuda.synchronize()
    ref = oracle_mod.device_resample(p.float().cpu().numpy(), q.cpu().numpy(), n.cpu().numpy(), u.cpu().numpy(), gamma,
                                     threads=8)
    tok = out["token"].cpu().numpy()
    # both sides add V float64 terms, in different orders: V * 2^-53 relative each
    bad = (tok != ref["token"]) & ~(ref["margin_cdf"] < V * 2.0 ** -52)
    assert not bad.any(), (np.nonzero(bad)[0][:8], tok[bad][:8], ref["token"][bad][:8])
    assert (out["flags"].cpu().numpy().astype(np.uint32) == ref["flags"]).all()


@pytest.mark.parametrize("Bn,V", [(5, 3000), (3, 20011), (40, 70001), (4, 300001), (4, 1100001), (120, 15001), (700, 4200), (4, 100003)])
def test_fallback_and_invalid_lengths(B, oracle_mod, Bn, V):
    """No residual mass (p == q): drawn from p; lengths outside [0, gamma] and rows without mass: token -1; one
    cluster per sequence, in turns, and the two-kernel path."""
    gamma = 2
    gen = torch.Generator(device="cuda").manual_seed(V)
    p = torch.softmax(2.0 * torch.randn(Bn, V, generator=gen, device="cuda"), dim=-1)
    q = p.view(Bn, 1, V).repeat(1, gamma, 1).contiguous()
    n = (torch.arange(Bn, device="cuda") % (gamma + 1)).to(torch.int32)
    n[0], n[1] = -1, gamma + 1
    p[2] = 0.0
    u = torch.rand(Bn, generator=gen, device="cuda").clamp_(max=1.0 - 2.0 ** -24)
    out = B.dssd_device_resample(p, q, n, u, gamma)
    torch.cuda.synchronize()
    ref = oracle_mod.device_resample(p.cpu().numpy(), q.cpu().numpy(), n.cpu().numpy(), u.cpu().numpy(), gamma)
    near = ref["margin_cdf"] < V * 2.0 ** -52  # V float64 additions in another order
    assert ((out["token"].cpu().numpy() == ref["token"]) | near).all()
    assert (out["flags"].cpu().numpy().astype(np.uint32) == ref["flags"]).all()


@pytest.mark.parametrize("Bn,V", [(130, 15000), (500, 9001)])
def test_rejected_sequences_only_in_turns(B, Bn, V):
    gamma = 2
    gen = torch.Generator(device="cuda").manual_seed(V)
    p = torch.softmax(2.0 * torch.randn(Bn, V, generator=gen, device="cuda"), dim=-1)
    q = torch.softmax(2.0 * torch.randn(Bn, gamma, V, generator=gen, device="cuda"), dim=-1)
    n = (torch.arange(Bn, device="cuda") % (gamma + 1)).to(torch.int32)
    u = torch.rand(Bn, generator=gen, device="cuda").clamp_(max=1.0 - 2.0 ** -24)
    full = B.dssd_device_resample(p, q, n, u, gamma)
    some = {"token": torch.full_like(n, 77), "flags": torch.full_like(n, 88)}
    B.dssd_device_resample_rejected(p, q, n, u, gamma, out=some)
    torch.cuda.synchronize()
    bonus = n == gamma
    assert (some["token"][bonus] == 77).all() and (some["flags"][bonus] == 88).all()
    assert torch.equal(some["token"][~bonus], full["token"][~bonus]) and torch.equal(some["flags"][~bonus], full["flags"][~bonus])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [20000, 20001])
def test_fused_draw_in_turns(B, V, dtype):
    """The draw straight from the logits, in turns, against the draw from the row that the edge writes (the same float32
    values and the same float64 sums)."""
    Bn, gamma, T = 150, 16, 0.9
    gen = torch.Generator(device="cuda").manual_seed(V)
    tl = (3.0 * torch.randn(Bn, gamma + 1, V, generator=gen, device="cuda")).to(dtype)
    q = torch.softmax(tl[:, :gamma].float() / T + 0.1 * torch.randn(Bn, gamma, V, generator=gen, device="cuda"), dim=-1)
    x = torch.multinomial(q.view(-1, V), 1, generator=gen).view(Bn, gamma)
    q_tok = torch.gather(q, 2, x.unsqueeze(2)).squeeze(2).contiguous()
    x = x.to(torch.int32)
    u = torch.rand(Bn, gamma, generator=gen, device="cuda")
    u_rs = torch.rand(Bn, generator=gen, device="cuda").clamp_(max=1.0 - 2.0 ** -24)
    ev = B.dssd_edge_verify(tl, x, q_tok, u, T)
    rs = B.dssd_device_resample(ev["p_row"], q, ev["accept_len"], u_rs, gamma)
    got = B.dssd_dsd_verify(tl, q, x, u, u_rs, T)
    torch.cuda.synchronize()
    assert torch.equal(got["accept_len"], ev["accept_len"]) and torch.equal(got["token"], rs["token"])
    assert torch.equal(got["rs_flags"], rs["flags"])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [20000, 20001])
def test_bonus_tokens_in_turns(B, V, dtype):
    """The bonus tokens drawn straight from the logits, in turns (more positions than the edge's one launch takes), against the draw
    from the rows that the edge writes; the others keep -1."""
    Bn, gamma, T = 60, 32, 0.9
    gen = torch.Generator(device="cuda").manual_seed(V)
    tl = (3.0 * torch.randn(Bn, gamma + 1, V, generator=gen, device="cuda")).to(dtype)
    x = torch.randint(0, V, (Bn, gamma), generator=gen, device="cuda", dtype=torch.int32)
    half = torch.full((Bn, gamma), 0.5, device="cuda")
    u = torch.zeros(Bn, gamma, device="cuda")  # accepted
    u[::3, 5] = 0.999
    u_rs = torch.rand(Bn, generator=gen, device="cuda").clamp_(max=1.0 - 2.0 ** -24)
    ev = B.dssd_edge_verify(tl, x, half, u, T)
    rs = B.dssd_device_resample(ev["p_row"], torch.zeros(Bn, gamma, V, device="cuda"), ev["accept_len"], u_rs, gamma)
    got = B.dssd_edge_verify_bonus(tl, x, half, u, u_rs, T)
    torch.cuda.synchronize()
    full = ev["accept_len"] == gamma
    assert torch.equal(got["accept_len"], ev["accept_len"]) and 0 < full.sum() < Bn
    assert torch.equal(got["token"][full], rs["token"][full]) and (got["token"][~full] == -1).all()
    assert torch.equal(got["token_flags"][full], rs["flags"][full]) and (got["token_flags"][~full] == 0).all()
