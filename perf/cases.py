"""Performance cases of the verification round: what a user of this library has it do.

A pass is one verification round of a batch through the Python entry points, with the output
buffers and workspaces that a serving loop keeps (allocated once, handed to every call).  Inputs
follow the noise model of `dssd_inputs/generator.py` (Gaussian target logits over a Zipf(1.1) bias,
draft logits = target logits + noise, drafted tokens sampled from the draft rows), made on the GPU
from the seed.

Kinds of round:
  dense   dssd_edge_verify, then dssd_device_resample              (Algorithm 2)
  f16     the same with the downlink row in 16 bits per value
  bonus   dssd_edge_verify_bonus, then dssd_device_resample_rejected (bonus token drawn at the edge)
  fused   dssd_dsd_verify                                          (Algorithm 1: one server does both halves)
  topk    dssd_edge_verify_topk, then dssd_device_resample_topk    (the paper's top-k sampler)
  shard   one rank of a vocabulary-sharded edge: the five shard calls, with the other ranks'
          contributions to the two all-gathers already in place
  host    dssd_round_host on pinned host buffers, copies included
"""
from __future__ import annotations

import math
from typing import Dict

import torch

from paper_2507_12000_b200 import binding as B

# the largest round: logits and draft rows of B = 1024, gamma = 16, V = 50272 in float32
MAX_LOGIT_BYTES = 1024 * 17 * 50272 * 4
MAX_DRAFT_BYTES = 1024 * 16 * 50272 * 4
# a round on host buffers is bound by the bus: kept to what one small server handles at a time
MAX_HOST_BYTES = 16 << 20


def _case(kind: str, batch: int, gamma: int, vocab: int, dtype: str, temperature: float, sigma_d: float, k: int = 0,
          shards: int = 0, name: str = "") -> Dict:
    c = {"kind": kind, "B": batch, "gamma": gamma, "V": vocab, "dtype": dtype, "T": temperature, "sigma_d": sigma_d,
         "k": k, "shards": shards}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's own regime: one sequence, eight drafted tokens, an OPT-sized vocabulary; the
        # latency of a round is what the user waits for
        _case("dense", 1, 8, 50272, "f32", 1.0, 0.6, name="dense_B1_g8_V50272_f32"),
        # a small server: a few sequences, bf16 logits straight from the model
        _case("dense", 8, 4, 32000, "bf16", 1.0, 0.7, name="dense_B8_g4_V32000_bf16"),
        # an ordinary serving batch with long drafts that are often rejected
        _case("dense", 64, 8, 128256, "bf16", 0.8, 1.0, name="dense_B64_g8_V128256_bf16"),
        # a large serving batch, good draft model (the benchmark's default workload)
        _case("dense", 256, 4, 151936, "bf16", 0.7, 0.4, name="dense_B256_g4_V151936_bf16"),
        # the largest: float32 logits, the longest drafts
        _case("dense", 1024, 16, 50272, "f32", 1.0, 0.6, name="dense_B1024_g16_V50272_f32"),
        # 16-bit downlink with rows that start on no 16-byte boundary (odd vocabulary)
        _case("f16", 300, 4, 30011, "bf16", 0.7, 0.5, name="f16_B300_g4_V30011_bf16"),
        # Algorithm 2 as printed, short drafts that are mostly accepted: many bonus tokens
        _case("bonus", 128, 4, 50272, "f32", 1.0, 0.2, name="bonus_B128_g4_V50272_f32"),
        # co-located draft and target model: Algorithm 1 in one call, no row in memory
        _case("fused", 256, 4, 151936, "bf16", 0.7, 0.4, name="fused_B256_g4_V151936_bf16"),
        # the paper's sampler (top-k, k = 10, T = 1) for one sequence ...
        _case("topk", 1, 8, 50272, "f32", 1.0, 0.6, k=10, name="topk10_B1_g8_V50272_f32"),
        # ... and for a large batch
        _case("topk", 256, 4, 151936, "bf16", 0.7, 0.4, k=10, name="topk10_B256_g4_V151936_bf16"),
        # one of eight ranks of a tensor-parallel LM head
        _case("shard", 256, 4, 151936, "bf16", 0.7, 0.4, shards=8, name="shard8_B256_g4_V151936_bf16"),
        # the whole round on host buffers (a server whose model runs elsewhere)
        _case("host", 8, 4, 32000, "bf16", 1.0, 0.7, name="host_B8_g4_V32000_bf16"),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "f16", "bonus", "fused", "topk", "topk", "shard", "host"])
    while True:
        batch = _log_int(rng, 1, 1024)
        gamma = _log_int(rng, 1, 16)
        vocab = _log_int(rng, 1024, 160000)
        if rng.random() < 0.6:  # most vocabularies are padded to a multiple of 16, the others are odd sizes
            vocab = (vocab + 15) // 16 * 16
        dtype = rng.choice(["bf16", "f32"])
        esz = 2 if dtype == "bf16" else 4
        logit_bytes = batch * (gamma + 1) * vocab * esz
        draft_bytes = batch * gamma * vocab * 4
        if logit_bytes > MAX_LOGIT_BYTES or draft_bytes > MAX_DRAFT_BYTES:
            continue
        if kind == "host" and logit_bytes + draft_bytes > MAX_HOST_BYTES:
            continue
        break
    temperature = rng.choice([0.6, 0.7, 0.8, 1.0, 1.2])
    sigma_d = round(rng.uniform(0.2, 1.2), 2)
    k = rng.choice([1, 4, 10, 10, 20, 32]) if kind == "topk" else 0
    shards = rng.choice([2, 4, 8]) if kind == "shard" else 0
    return _case(kind, batch, gamma, vocab, dtype, temperature, sigma_d, k, shards)


# ---- inputs ----------------------------------------------------------------------------------


def _uniform(shape, gen) -> torch.Tensor:
    """Multiples of 2^-24 in [0, 1)."""
    return torch.randint(0, 1 << 24, shape, generator=gen, device="cuda").to(torch.float32) * 2.0 ** -24


def _inputs(case, seed: int) -> Dict[str, torch.Tensor]:
    nb, g, V, T, k = case["B"], case["gamma"], case["V"], case["T"], case["k"]
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    beta = -1.1 * torch.log1p(torch.randperm(V, generator=gen, device=dev).to(torch.float32))
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    d = {
        "target_logits": torch.empty(nb, g + 1, V, dtype=dt, device=dev),
        "draft_tokens": torch.empty(nb, g, dtype=torch.int32, device=dev),
        "draft_q_tok": torch.empty(nb, g, dtype=torch.float32, device=dev),
        "uniforms": _uniform((nb, g), gen),
        "uniforms_rs": _uniform((nb,), gen),
    }
    if k:
        d["q_idx"] = torch.empty(nb, g, k, dtype=torch.int32, device=dev)
        d["q_val"] = torch.empty(nb, g, k, dtype=torch.float32, device=dev)
    else:
        d["draft_q"] = torch.empty(nb, g, V, dtype=torch.float32, device=dev)
    ud = _uniform((nb, g, 1), gen)
    step = max(1, (1 << 26) // ((g + 1) * V))  # sequences at a time: a quarter of a GB of logits
    for b0 in range(0, nb, step):
        b1 = min(nb, b0 + step)
        tl = torch.randn(b1 - b0, g + 1, V, generator=gen, device=dev).mul_(3.0).add_(beta)
        d["target_logits"][b0:b1] = tl
        q = torch.randn(b1 - b0, g, V, generator=gen, device=dev).mul_(case["sigma_d"]).add_(tl[:, :g]).div_(T)
        del tl
        q = torch.softmax(q, dim=-1)
        if k:
            val, idx = torch.topk(q, k, dim=-1)
            q = val / val.sum(dim=-1, keepdim=True)
            d["q_idx"][b0:b1] = idx.to(torch.int32)
            d["q_val"][b0:b1] = q
        else:
            d["draft_q"][b0:b1] = q
        cdf = torch.cumsum(q, dim=-1)
        at = torch.searchsorted(cdf, ud[b0:b1] * cdf[:, :, -1:], right=True).clamp_(max=q.shape[-1] - 1)
        d["draft_q_tok"][b0:b1] = torch.gather(q, 2, at).squeeze(2)
        d["draft_tokens"][b0:b1] = (torch.gather(idx, 2, at) if k else at).squeeze(2).to(torch.int32)
    return d


def _ints(*names, n: int) -> Dict[str, torch.Tensor]:
    return {name: torch.zeros(n, dtype=torch.int32, device="cuda") for name in names}


def _workspace(nbytes: int) -> torch.Tensor:
    return torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")


def _shard_bounds(V: int, G: int):
    """Contiguous slices of nearly equal size, multiples of 16 entries where the vocabulary allows it."""
    unit = 16 if V >= 64 * G else 1
    per = (V + G * unit - 1) // (G * unit) * unit
    cuts = [min(V, i * per) for i in range(G)] + [V]
    return [(cuts[i], cuts[i + 1]) for i in range(G)]


def _prepare_shard(case, d) -> Dict:
    """Rank g's slices and buffers; the other ranks' rows of the two gathered arrays are what those
    ranks would have sent."""
    nb, gamma, V, T, G = case["B"], case["gamma"], case["V"], case["T"], case["shards"]
    bounds = _shard_bounds(V, G)
    g = G // 2
    s = {
        "g": g, "v_begin": bounds[g][0],
        "part_ref": torch.empty(G, nb, gamma + 1, device="cuda"),
        "part_sum": torch.empty(G, nb, gamma + 1, dtype=torch.float64, device="cuda"),
        "tok_logit": torch.empty(G, nb, gamma, device="cuda"),
        "mass": torch.empty(G, nb, 2, dtype=torch.float64, device="cuda"),
    }
    tl, dq = d.pop("target_logits"), d.pop("draft_q")
    for h, (a, b) in enumerate(bounds):
        B.dssd_edge_partial(tl[:, :, a:b], d["draft_tokens"], a, T, out=_slot(s, h))
    ev = B.dssd_edge_combine(s["part_ref"], s["part_sum"], s["tok_logit"], d["draft_tokens"], d["draft_q_tok"],
                             d["uniforms"], T, V)
    for h, (a, b) in enumerate(bounds):
        row = B.dssd_edge_emit_shard(tl[:, :, a:b], ev["accept_len"], ev["row_scale"], T)
        B.dssd_resample_shard_mass(row, dq[:, :, a:b], ev["accept_len"], gamma, out=s["mass"][h])
    a, b = bounds[g]
    s["logits"] = tl[:, :, a:b].contiguous()
    s["draft_q"] = dq[:, :, a:b].contiguous()
    s["part_out"] = _slot(s, g)
    s["ev_out"] = ev
    s["row_out"] = torch.empty(nb, b - a, device="cuda")
    s["rs_out"] = _ints("token", "flags", n=nb)
    s["ws_e"] = _workspace(B.dssd_edge_partial_workspace_bytes(nb, gamma, b - a))
    s["ws_r"] = _workspace(B.dssd_resample_shard_workspace_bytes(nb, gamma, b - a))
    return s


def _slot(s, h: int) -> Dict[str, torch.Tensor]:
    return {"part_ref": s["part_ref"][h], "part_sum": s["part_sum"][h], "tok_logit": s["tok_logit"][h]}


def prepare(case, seed):
    nb, gamma, V, k, kind = case["B"], case["gamma"], case["V"], case["k"], case["kind"]
    d = _inputs(case, seed)
    s = {"case": dict(case), "d": d}
    if kind == "host":
        s["host"] = {name: t.cpu().pin_memory() for name, t in d.items()}
        s["d"] = {}
        s["arena"] = _workspace(B.dssd_round_host_arena_bytes(
            nb, gamma, V, B.DSSD_BF16 if case["dtype"] == "bf16" else B.DSSD_F32))
        s["out"] = {name: torch.zeros(nb, dtype=torch.int32).pin_memory()
                    for name in ("accept_len", "token", "edge_flags", "rs_flags")}
        return s
    if kind == "shard":
        s.update(_prepare_shard(case, d))
        return s
    if kind == "fused":
        s["out"] = _ints("accept_len", "token", "edge_flags", "rs_flags", n=nb)
        s["ws"] = _workspace(B.dssd_dsd_verify_workspace_bytes(nb, gamma, V))
        return s
    ev = _ints("accept_len", "flags", n=nb)
    ev["p_tok"] = torch.zeros(nb, gamma, device="cuda")
    if kind == "topk":
        ev["p_idx"] = torch.zeros(nb, k, dtype=torch.int32, device="cuda")
        ev["p_val"] = torch.zeros(nb, k, device="cuda")
        s["ws_e"] = _workspace(B.dssd_edge_verify_topk_workspace_bytes(nb, gamma, V, k))
    else:
        ev["lse"] = torch.zeros(nb, gamma + 1, device="cuda")
        ev["p_row"] = torch.zeros(nb, V, dtype=torch.float16 if kind == "f16" else torch.float32, device="cuda")
        s["ws_e"] = _workspace(B.dssd_edge_verify_bonus_workspace_bytes(nb, gamma, V) if kind == "bonus"
                               else B.dssd_edge_verify_workspace_bytes(nb, gamma, V))
        s["ws_r"] = _workspace(B.dssd_device_resample_workspace_bytes(nb, gamma, V))
    if kind == "bonus":
        ev.update(_ints("token", "token_flags", n=nb))
        s["rs_out"] = {"token": ev["token"], "flags": ev["token_flags"]}
    else:
        s["rs_out"] = _ints("token", "flags", n=nb)
    s["ev_out"] = ev
    return s


# ---- one pass --------------------------------------------------------------------------------


def run(state):
    case, d = state["case"], state["d"]
    kind, gamma, T = case["kind"], case["gamma"], case["T"]
    if kind == "host":
        return B.dssd_round_host(state["host"], T, state["arena"], out=state["out"])
    if kind == "fused":
        return B.dssd_dsd_verify(d["target_logits"], d["draft_q"], d["draft_tokens"], d["uniforms"], d["uniforms_rs"], T,
                                 out=state["out"], workspace=state["ws"])
    if kind == "shard":
        part = B.dssd_edge_partial(state["logits"], d["draft_tokens"], state["v_begin"], T, out=state["part_out"],
                                   workspace=state["ws_e"])
        ev = B.dssd_edge_combine(state["part_ref"], state["part_sum"], state["tok_logit"], d["draft_tokens"],
                                 d["draft_q_tok"], d["uniforms"], T, case["V"], out=state["ev_out"])
        row = B.dssd_edge_emit_shard(state["logits"], ev["accept_len"], ev["row_scale"], T, out=state["row_out"])
        mass, ws = B.dssd_resample_shard_mass(row, state["draft_q"], ev["accept_len"], gamma, out=state["mass"][state["g"]],
                                              workspace=state["ws_r"])
        rs = B.dssd_resample_shard_draw(state["mass"], state["g"], state["v_begin"], row, state["draft_q"],
                                        ev["accept_len"], d["uniforms_rs"], gamma, ws, out=state["rs_out"])
        return {"part": part, "edge": ev, "row": row, "mass": mass, "draw": rs}
    if kind == "topk":
        ev = B.dssd_edge_verify_topk(d["target_logits"], d["draft_tokens"], d["draft_q_tok"], d["uniforms"], T, case["k"],
                                     out=state["ev_out"], workspace=state["ws_e"])
        rs = B.dssd_device_resample_topk(ev["p_idx"], ev["p_val"], d["q_idx"], d["q_val"], ev["accept_len"],
                                         d["uniforms_rs"], gamma, out=state["rs_out"])
        return {"edge": ev, "draw": rs}
    if kind == "bonus":
        ev = B.dssd_edge_verify_bonus(d["target_logits"], d["draft_tokens"], d["draft_q_tok"], d["uniforms"],
                                      d["uniforms_rs"], T, out=state["ev_out"], workspace=state["ws_e"])
        rs = B.dssd_device_resample_rejected(ev["p_row"], d["draft_q"], ev["accept_len"], d["uniforms_rs"], gamma,
                                             out=state["rs_out"], workspace=state["ws_r"])
        return {"edge": ev, "draw": rs}
    ev = B.dssd_edge_verify(d["target_logits"], d["draft_tokens"], d["draft_q_tok"], d["uniforms"], T, out=state["ev_out"],
                            workspace=state["ws_e"], payload="f16" if kind == "f16" else "f32")
    rs = B.dssd_device_resample(ev["p_row"], d["draft_q"], ev["accept_len"], d["uniforms_rs"], gamma, out=state["rs_out"],
                                workspace=state["ws_r"])
    return {"edge": ev, "draw": rs}


# ---- what a pass cannot do without -----------------------------------------------------------


def work(case):
    nb, g, V, kind = case["B"], case["gamma"], case["V"], case["kind"]
    esz = 2 if case["dtype"] == "bf16" else 4
    # per-token acceptance of the noise model and the share of sequences with a rejection
    alpha = max(0.3, 1.0 - 0.35 * case["sigma_d"] / math.sqrt(case["T"]))
    rejected = 1.0 - alpha ** g
    if kind == "shard":
        V = _shard_bounds(V, case["shards"])[case["shards"] // 2]
        V = V[1] - V[0]
    logits = nb * (g + 1) * V * esz
    row = {"dense": 8.0, "shard": 8.0, "f16": 4.0, "bonus": 8.0 * rejected}.get(kind, 0.0)  # written, then read
    q_row = 0.0 if kind == "topk" else 4.0 * rejected
    return {"bytes": logits + nb * V * (row + q_row), "flops": 4.0 * nb * (g + 1) * V}


def tolerance(case):
    if case["kind"] == "topk":
        # float64 throughout, one rounding to float32 (measured against float64: 3e-8, largest 6e-8)
        return {"rel": 2e-7, "max": 5e-7}
    # Whole values (lengths, tokens, flags) may differ where a uniform falls on a step of a distribution.
    if case["kind"] == "f16":
        # a value within float32 rounding of a binary16 rounding boundary moves by one binary16
        # unit, 2^-11 to 2^-10 of itself; the row's largest entry may be one of them
        return {"rel": 5e-4, "max": 1e-3, "differ": 0.01}
    # Probabilities formed in float32: scaling by log2(e) / T, one exponential, float32 sums.  Measured
    # against float64: 1.1e-7, largest 6e-7; a residual mass Z is relative to 1 and so off by 1 / Z more.
    return {"rel": 2e-6, "max": 1e-5, "differ": 0.01}
