"""The rounds on host buffers, pinned (read and written over the bus by the kernels), pageable (copied) and
mixed, short arrays and arrays beyond what the staging kernel takes: the same results as the device calls."""
import pytest
import torch

import dssd_inputs as di
from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_12000_b200 import binding

    return binding


def _host(g, pin):
    out = {}
    for i, (k, v) in enumerate(g.items()):
        t = v.cpu()
        out[k] = t.pin_memory() if pin == "all" or (pin == "some" and i % 2) else t
    return out


@pytest.mark.parametrize("pin", ["all", "none", "some"])
@pytest.mark.parametrize("Bn,gamma,V,dtype", [(3, 2, 4001, "bf16"), (40, 3, 9000, "f32"), (9, 0, 3000, "f32"), (6000, 3, 64, "bf16")])
def test_dense_round(B, pin, Bn, gamma, V, dtype):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.5, seed=Bn + V)
    g = to_device(di.generate(w, threads=8))
    ev = B.dssd_edge_verify(g["target_logits"], g["draft_tokens"], g["draft_q_tok"], g["uniforms"], w.temperature)
    rs = B.dssd_device_resample(ev["p_row"], g["draft_q"], ev["accept_len"], g["uniforms_rs"], gamma)
    arena = torch.full((B.dssd_round_host_arena_bytes(Bn, gamma, V, B.DSSD_BF16 if dtype == "bf16" else B.DSSD_F32),), 0x5A,
                       dtype=torch.uint8, device="cuda")
    out = {k: torch.zeros(Bn, dtype=torch.int32) for k in ("accept_len", "token", "edge_flags", "rs_flags")}
    out["p_row"] = torch.zeros(Bn, V)
    out = _host(out, pin)
    got = B.dssd_round_host(_host(g, pin), w.temperature, arena, out=out)
    n_at_return = got["accept_len"].clone()
    torch.cuda.synchronize()
    assert torch.equal(n_at_return, ev["accept_len"].cpu())  # final when the call returns
    assert torch.equal(got["token"], rs["token"].cpu()) and torch.equal(got["p_row"], ev["p_row"].cpu())
    assert torch.equal(got["edge_flags"], ev["flags"].cpu()) and torch.equal(got["rs_flags"], rs["flags"].cpu())


@pytest.mark.parametrize("pin", ["all", "none", "some"])
def test_topk_round(B, pin):
    k = 10
    w = di.custom(B=20, gamma=3, V=9001, dtype="bf16", temperature=0.9, sigma_d=0.5, seed=3)
    g = to_device(di.generate_topk(w, k, threads=8))
    ev = B.dssd_edge_verify_topk(g["target_logits"], g["draft_tokens"], g["draft_q_tok"], g["uniforms"], w.temperature, k)
    rs = B.dssd_device_resample_topk(ev["p_idx"], ev["p_val"], g["q_idx"], g["q_val"], ev["accept_len"], g["uniforms_rs"], w.gamma)
    arena = torch.full((B.dssd_round_host_topk_arena_bytes(w.B, w.gamma, w.V, k, B.DSSD_BF16),), 0x5A, dtype=torch.uint8, device="cuda")
    out = {n: torch.zeros(w.B, dtype=torch.int32) for n in ("accept_len", "token", "edge_flags", "rs_flags")}
    out["p_idx"], out["p_val"] = torch.zeros(w.B, k, dtype=torch.int32), torch.zeros(w.B, k)
    got = B.dssd_round_host_topk(_host(g, pin), w.temperature, k, arena, out=_host(out, pin))
    torch.cuda.synchronize()
    for name, want in (("accept_len", ev["accept_len"]), ("token", rs["token"]), ("edge_flags", ev["flags"]), ("rs_flags", rs["flags"]),
                       ("p_idx", ev["p_idx"]), ("p_val", ev["p_val"])):
        assert torch.equal(got[name], want.cpu()), name


@pytest.mark.parametrize("pages", [[(0, 3), (9, 12)], [(0, 5), (5, 12)], [(0, 12)], [(2, 12)]])
def test_draft_rows_pinned_in_pieces(B, pages):
    """draft_q of 12 rows of one page each, of which only some pages are registered: read in place where all are (in one range or in
    two that follow one another), else copied row by row, also where its first and last bytes are pinned."""
    Bn, gamma, V = 3, 4, 1024
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype="f32", temperature=0.9, sigma_d=1.0, seed=8)
    g = to_device(di.generate(w, threads=8))
    arena = torch.empty(B.dssd_round_host_arena_bytes(Bn, gamma, V, B.DSSD_F32), dtype=torch.uint8, device="cuda")
    host = _host(g, "all")
    raw = torch.empty(13 * 4096, dtype=torch.uint8)
    at = -raw.data_ptr() % 4096
    host["draft_q"] = raw[at:at + 12 * 4096].view(torch.float32).view(Bn, gamma, V).copy_(host["draft_q"])
    base, rt = host["draft_q"].data_ptr(), torch.cuda.cudart()
    for a, b in pages:
        assert int(rt.cudaHostRegister(base + a * 4096, (b - a) * 4096, 0)) == 0
    try:
        for n_at in range(gamma + 1):  # the rejection at every position in turn
            host["uniforms"].fill_(0.0)
            host["uniforms"][:, n_at:] = 1.0
            n = torch.full((Bn,), n_at, dtype=torch.int32, device="cuda")
            ev = B.dssd_edge_verify(g["target_logits"], g["draft_tokens"], g["draft_q_tok"], host["uniforms"].cuda(), w.temperature)
            assert torch.equal(ev["accept_len"], n)
            rs = B.dssd_device_resample(ev["p_row"], g["draft_q"], n, g["uniforms_rs"], gamma)
            got = B.dssd_round_host(host, w.temperature, arena)
            torch.cuda.synchronize()
            assert torch.equal(got["accept_len"], n.cpu()) and torch.equal(got["token"], rs["token"].cpu())
            assert torch.equal(got["rs_flags"], rs["flags"].cpu())
    finally:
        for a, _ in pages:
            assert int(rt.cudaHostUnregister(base + a * 4096)) == 0


@pytest.mark.parametrize("Bn,gamma,V,dtype,offset", [
    (1, 0, 5, "bf16", 0),       # shorter than one vector
    (5, 1, 4096, "bf16", 0),    # whole CTAs of the kernel that reads them over the bus
    (3, 1, 8193, "bf16", 0),    # six whole CTAs and twelve bytes
    (1, 0, 8191, "bf16", 0),    # a vector less than a whole CTA, and fourteen bytes
    (1, 0, 8201, "bf16", 0),    # a vector more, and two bytes
    (1, 0, 10595, "bf16", 0),   # 300 vectors more, within a thread's second load, and six bytes
    (1, 0, 4099, "f32", 0),     # a whole CTA and twelve bytes, of the other type
    (3, 1, 8193, "bf16", 3),    # not on a boundary of 16 bytes: copied
    (2, 1, 262144, "f32", 0),   # the longest logits that are read over the bus ...
    (2, 1, 262145, "f32", 0),   # ... and longer ones
])
def test_pinned_logits(B, Bn, gamma, V, dtype, offset):
    w = di.custom(B=Bn, gamma=gamma, V=V, dtype=dtype, temperature=0.9, sigma_d=0.5, seed=V + offset)
    g = to_device(di.generate(w, threads=8))
    ev = B.dssd_edge_verify(g["target_logits"], g["draft_tokens"], g["draft_q_tok"], g["uniforms"], w.temperature)
    rs = B.dssd_device_resample(ev["p_row"], g["draft_q"], ev["accept_len"], g["uniforms_rs"], gamma)
    host = _host(g, "all")
    tl = host["target_logits"]
    host["target_logits"] = torch.empty(tl.numel() + offset, dtype=tl.dtype, pin_memory=True)[offset:].view(tl.shape).copy_(tl)
    arena = torch.full((B.dssd_round_host_arena_bytes(Bn, gamma, V, B.DSSD_BF16 if dtype == "bf16" else B.DSSD_F32),), 0x5A,
                       dtype=torch.uint8, device="cuda")
    out = {"p_row": torch.zeros(Bn, V)}
    out.update({k: torch.zeros(Bn, dtype=torch.int32) for k in ("accept_len", "token", "edge_flags", "rs_flags")})
    got = B.dssd_round_host(host, w.temperature, arena, out=out)
    torch.cuda.synchronize()
    assert torch.equal(got["accept_len"], ev["accept_len"].cpu()) and torch.equal(got["token"], rs["token"].cpu())
    assert torch.equal(got["p_row"], ev["p_row"].cpu())
