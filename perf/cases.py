"""The work a user of this library has it do, as cases that can be timed.

One speculative step verifies gamma drafted tokens of every sequence: the mask
metadata, one attention call per layer over the paged K/V cache, the
acceptance of the drafts over the logits, and the commit of the accepted K/V.
The cases are the layers' attention calls over the range of batches, prefix
lengths, draft lengths, page sizes and data types the library is used with,
the two acceptance rules, and two whole steps.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  what a program holds before the call: inputs, block
                       tables, mask metadata, workspaces, a captured step
  run(state)           one pass through the public entry points
  work(case)           bytes and flops one pass cannot do without
  exact(case, seed)    run()'s floating results in 64 bits, by plain torch
"""
from __future__ import annotations

import dataclasses
import math

import torch

from paper_2606_02544_gb300 import inputs, simsd
from paper_2606_02544_gb300.step import VerifyStep

_SD = 1.0 / math.sqrt(128.0)  # scale of Q, K and V in the bf16 workloads
_THETA = 1.0e6                # RoPE base of the SDAR backbones
_VOCAB = 151936               # vocabulary of the SDAR models

# most work a drawn case may ask for (the largest listed cases do more)
_MAX_KV_BYTES = 1.2e9
_MAX_F32_FLOPS = 2.0e10
_MAX_LOGIT_BYTES = 6.0e8


def _attention(name, dtype, Bt, Hq, Hkv, d, gamma, lo, hi, page=64, rope=False, order="identity"):
    return {"name": name, "kind": "attention", "dtype": dtype, "Bt": Bt, "Hq": Hq, "Hkv": Hkv, "d": d,
            "gamma": gamma, "lo": lo, "hi": hi, "page": page, "rope": rope, "order": order}


def _step(name, dtype, Bt, Hq, Hkv, d, gamma, lo, hi, layers, vocab, p_agree, page=64, rope=False,
          order="identity"):
    return {"name": name, "kind": "step", "dtype": dtype, "Bt": Bt, "Hq": Hq, "Hkv": Hkv, "d": d, "gamma": gamma,
            "lo": lo, "hi": hi, "page": page, "rope": rope, "order": order, "layers": layers, "vocab": vocab,
            "p_agree": p_agree}


def listed():
    return [
        # the smallest call: a whole fp32 step of one short sequence, where
        # the launches and one memory latency per kernel are everything
        _step("step_tiny_fp32", "f32", 1, 2, 1, 64, 4, 128, 128, 1, 1024, 0.7),
        # a whole step of a small serving batch through all 36 layers, the
        # way a decoding loop runs it: captured once, queries and new keys
        # rotated inside, drafts in confidence order
        _step("step_sdar8b_b8_rope", "bf16", 8, 32, 8, 128, 8, 512, 2048, 36, _VOCAB, 0.6, rope=True,
              order="permuted"),
        # one layer of a small model at a small batch (latency)
        _attention("attn_sdar1.7b_b8", "bf16", 8, 16, 8, 128, 4, 512, 1024),
        # one layer, an ordinary serving batch with equal prefixes
        _attention("attn_sdar4b_b32", "bf16", 32, 32, 8, 128, 8, 4096, 4096),
        # one layer of the large ragged batch (the headline workload's layer)
        _attention("attn_sdar8b_b64", "bf16", 64, 32, 8, 128, 16, 2048, 8192),
        # one user with a long context: few units, the prefix split over the GPU
        _attention("attn_sdar8b_b1_long", "bf16", 1, 32, 8, 128, 8, 32768, 32768),
        # long drafts: 256 query rows per KV head, near the compute ridge
        _attention("attn_sdar8b_b32_draft32", "bf16", 32, 32, 8, 128, 32, 2048, 8192),
        # small pages, RoPE in the call, blocks only partly drafted: the
        # options of an engine with its own page size, at a ragged batch
        _attention("attn_sdar8b_b19_page16_rope", "bf16", 19, 32, 8, 128, 7, 190, 3000, page=16, rope=True,
                   order="partial"),
        # the paper's own precision, at the small model's layer
        _attention("attn_sdar1.7b_b8_fp32", "f32", 8, 16, 8, 128, 4, 512, 1024),
        # greedy acceptance of the large batch: the vocabulary-wide argmax
        {"name": "accept_b64", "kind": "accept", "Bt": 64, "gamma": 16, "vocab": _VOCAB, "p_agree": 0.8},
        # greedy acceptance with a vocabulary that is no multiple of 4 (an
        # added token): rows start off the 16-byte grid
        {"name": "accept_b16_odd_vocab", "kind": "accept", "Bt": 16, "gamma": 8, "vocab": 50001, "p_agree": 0.6},
        # stochastic acceptance at a small batch (target and draft logits)
        {"name": "accept_sampled_b8", "kind": "sampled", "Bt": 8, "gamma": 8, "vocab": _VOCAB, "eta": 0.5,
         "temperature": 0.8},
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _prefixes(rng, lo, hi):
    top = _logint(rng, lo, hi)
    return rng.choice([top, max(1, int(top * rng.uniform(0.2, 1.0)))]), top


def draw(rng):
    kind = rng.choices(["attention", "attention_f32", "step", "accept", "sampled"], [8, 2, 2, 3, 3])[0]
    if kind == "attention":
        while True:
            Hq = rng.choice([16, 32, 32])
            gamma = _logint(rng, 4, 32)
            Bt = _logint(rng, 1, 128)
            lo, hi = _prefixes(rng, 128, 32768)
            if Bt * hi * 8 * 128 * 4 <= _MAX_KV_BYTES:
                break
        c = _attention("", "bf16", Bt, Hq, 8, 128, gamma, lo, hi, rng.choice([16, 32, 64, 64, 128]),
                       rng.random() < 0.5, rng.choice(["identity", "permuted", "partial"]))
    elif kind == "attention_f32":
        while True:
            d = rng.choice([64, 128, 128])
            Hq, Hkv = rng.choice([(2, 1), (16, 8), (32, 8)])
            gamma = _logint(rng, 4, 32)
            Bt = _logint(rng, 1, 32)
            lo, hi = _prefixes(rng, 128, 4096)
            if 4.0 * d * Hq * 2 * gamma * Bt * hi <= _MAX_F32_FLOPS:
                break
        c = _attention("", "f32", Bt, Hq, Hkv, d, gamma, lo, hi, rng.choice([16, 64, 64, 128]), rng.random() < 0.5,
                       rng.choice(["identity", "permuted", "partial"]))
    elif kind == "step":
        while True:
            layers = _logint(rng, 1, 36)
            Bt = _logint(rng, 1, 32)
            lo, hi = _prefixes(rng, 128, 4096)
            if layers * Bt * hi * 8 * 128 * 4 <= _MAX_KV_BYTES:
                break
        c = _step("", "bf16", Bt, rng.choice([16, 32]), 8, 128, _logint(rng, 4, 16), lo, hi, layers,
                  rng.choice([_VOCAB, _logint(rng, 1000, _VOCAB)]), rng.uniform(0.3, 0.9), rng.choice([16, 64]),
                  rng.random() < 0.5, rng.choice(["identity", "permuted"]))
    elif kind == "accept":
        while True:
            Bt, gamma = _logint(rng, 1, 128), _logint(rng, 4, 32)
            vocab = rng.choice([_VOCAB, _VOCAB, _logint(rng, 1000, _VOCAB)])
            if Bt * (gamma + 1) * vocab * 4 <= _MAX_LOGIT_BYTES:
                break
        c = {"kind": "accept", "Bt": Bt, "gamma": gamma, "vocab": vocab, "p_agree": rng.uniform(0.3, 0.9)}
    else:
        while True:
            Bt, gamma = _logint(rng, 1, 64), _logint(rng, 4, 32)
            vocab = rng.choice([_VOCAB, _VOCAB, _logint(rng, 1000, _VOCAB)])
            if Bt * (2 * gamma + 1) * vocab * 4 <= _MAX_LOGIT_BYTES:
                break
        c = {"kind": "sampled", "Bt": Bt, "gamma": gamma, "vocab": vocab, "eta": rng.uniform(0.1, 1.0),
             "temperature": rng.uniform(0.5, 1.2)}
    c.pop("name", None)
    return c


# --------------------------------------------------------------- preparation

def _workload(c, seed):
    std, sigma = (1.0, 1.0) if c["dtype"] == "f32" else (_SD, 2.0)
    return inputs.Workload("case", c["dtype"], c["Bt"], c["Hq"], c["Hkv"], c["d"], c["gamma"], (c["lo"], c["hi"]),
                           c.get("layers", 1), c.get("vocab", 1), c.get("p_agree", 0.0), std, sigma, seed, c["page"])


def _prefix_lengths(c, seed):
    """Lengths spread evenly over [lo, hi], in an order drawn from the seed
    (so that the page pool has the same size for every seed)."""
    n = [c["lo"] + int((c["hi"] - c["lo"]) * (i + 0.5) / c["Bt"]) for i in range(c["Bt"])]
    return [n[i] for i in torch.randperm(c["Bt"], generator=torch.Generator().manual_seed(seed)).tolist()]


def _step_inputs(c, seed):
    si = inputs.make_step_inputs(_workload(c, seed), device="cuda", random_step_map=c["order"] == "permuted",
                                 prefix_override=_prefix_lengths(c, seed), with_logits=c["kind"] == "step")
    if c["order"] == "partial":
        # blocks with fewer drafts than positions, some decoded already
        si = dataclasses.replace(si, step_map=inputs.block_step_maps(c["Bt"], c["gamma"], seed + 3).cuda())
    return si


def _i32(*shape):
    return torch.empty(*shape, dtype=torch.int32, device="cuda")


def _workspace(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda") if nbytes > 0 else None


def _logits(rows, vocab, seed, sigma=2.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*rows, vocab, generator=g, device="cuda").mul_(sigma), g


def prepare(case, seed):
    c = case
    if c["kind"] == "step":
        # buffers of the step and its captured graph
        st = VerifyStep(_step_inputs(c, seed), rope_theta=_THETA if c["rope"] else 0.0)
        st.capture(time_attention=False)
        return {"kind": "step", "step": st}
    if c["kind"] == "attention":
        si = _step_inputs(c, seed)
        w = si.w
        s = {"kind": "attention", "q": si.q[0], "k_new": si.k_new[0], "v_new": si.v_new[0], "k_cache": si.k_cache[0],
             "v_cache": si.v_cache[0], "block_table": si.block_table, "prefix_len": si.prefix_len,
             "tau": _i32(w.Bt, w.S), "section": torch.empty(w.Bt, w.S, dtype=torch.uint8, device="cuda"),
             "err": torch.zeros(1, dtype=torch.int32, device="cuda"), "out": torch.empty_like(si.q[0]),
             "rope_theta": _THETA if c["rope"] else 0.0}
        pos = _i32(w.Bt, w.S)
        # a step's mask metadata serves all of its layers
        simsd.simsd_build_mask(si.step_map, si.prefix_len, w.gamma, s["tau"], s["section"], pos, err_word=s["err"])
        s["rope_pos"] = pos if c["rope"] else None
        s["workspace"] = _workspace(simsd.simsd_verify_workspace_bytes(
            simsd.SIMSD_F32 if c["dtype"] == "f32" else simsd.SIMSD_BF16, w.Bt, w.gamma, w.Hq, w.Hkv, w.d,
            si.block_table.shape[1], w.page_size))
        return s
    Bt, gamma, V = c["Bt"], c["gamma"], c["vocab"]
    s = {"kind": c["kind"], "accepted": _i32(Bt), "tokens": _i32(Bt, gamma + 1),
         "err": torch.zeros(1, dtype=torch.int32, device="cuda")}
    s["logits"], g = _logits((Bt, gamma + 1), V, seed)
    if c["kind"] == "accept":
        agree = torch.rand(Bt, gamma, generator=g, device="cuda") < c["p_agree"]
        other = torch.randint(0, V, (Bt, gamma), generator=g, device="cuda")
        s["draft"] = torch.where(agree, s["logits"][:, :gamma].argmax(dim=-1), other).to(torch.int32)
        s["argmax"] = _i32(Bt, gamma + 1)
        s["workspace"] = _workspace(simsd.simsd_accept_workspace_bytes(Bt, gamma, V))
        return s
    # the draft model's logits lie near the target's; each draft is drawn
    # from its softmax (Gumbel-max)
    s["temperature"] = c["temperature"]
    s["draft_logits"] = torch.randn(Bt, gamma, V, generator=g, device="cuda").mul_(2.0 * c["eta"])
    s["draft_logits"] += s["logits"][:, :gamma]
    s["draft"] = _i32(Bt, gamma)
    for b in range(Bt):
        u = torch.rand(gamma, V, generator=g, device="cuda").clamp_(1e-30, 1.0 - 1e-7)
        u = s["draft_logits"][b] / c["temperature"] - torch.log(-torch.log(u))
        s["draft"][b] = u.argmax(dim=-1)
    s["u_accept"] = torch.rand(Bt, gamma, generator=g, device="cuda")
    s["u_sample"] = torch.rand(Bt, generator=g, device="cuda")
    s["workspace"] = _workspace(simsd.simsd_accept_sampled_workspace_bytes(Bt, gamma, V))
    return s


def run(state):
    s = state
    if s["kind"] == "step":
        st = s["step"]
        st.replay()
        return {"out": st.out, "accepted": st.accepted_len, "tokens": st.out_tokens, "argmax": st.row_argmax,
                "prefix_len": st.n, "k_cache": st.si.k_cache, "v_cache": st.si.v_cache}
    if s["kind"] == "attention":
        simsd.simsd_verify_attention(s["q"], s["k_new"], s["v_new"], s["k_cache"], s["v_cache"], s["block_table"],
                                     s["prefix_len"], s["tau"], s["section"], s["out"], workspace=s["workspace"],
                                     err_word=s["err"], rope_pos=s["rope_pos"], rope_theta=s["rope_theta"])
        return {"out": s["out"]}
    if s["kind"] == "accept":
        simsd.simsd_accept_ws(s["logits"], s["draft"], s["accepted"], s["tokens"], s["workspace"],
                              row_argmax=s["argmax"], err_word=s["err"])
        return {"accepted": s["accepted"], "tokens": s["tokens"], "argmax": s["argmax"]}
    simsd.simsd_accept_sampled_ws(s["logits"], s["draft_logits"], s["draft"], s["u_accept"], s["u_sample"],
                                  s["accepted"], s["tokens"], s["workspace"], temperature=s["temperature"],
                                  err_word=s["err"])
    return {"accepted": s["accepted"], "tokens": s["tokens"]}


# ------------------------------------------------------------------ accounts

def work(case):
    c = case
    if c["kind"] in ("accept", "sampled"):
        rows = c["Bt"] * ((c["gamma"] + 1) + (c["gamma"] if c["kind"] == "sampled" else 0))
        return {"bytes": rows * c["vocab"] * 4.0, "flops": rows * c["vocab"] * 2.0}
    eb = 4 if c["dtype"] == "f32" else 2
    S, n = 2 * c["gamma"], c["Bt"] * 0.5 * (c["lo"] + c["hi"])
    layer = (n * c["Hkv"] * c["d"] * 2 + 2.0 * c["Bt"] * S * (c["Hq"] + c["Hkv"]) * c["d"]) * eb
    flops = 4.0 * c["d"] * c["Hq"] * S * (n + c["Bt"] * c["gamma"])
    if c["kind"] == "attention":
        return {"bytes": layer, "flops": flops}
    p, L = c["p_agree"], c["layers"]
    kept = c["Bt"] * sum(p ** k for k in range(1, c["gamma"] + 1))
    commit = 2.0 * kept * c["Hkv"] * c["d"] * eb  # K and V rows written (read by the attention already)
    return {"bytes": L * (layer + commit) + c["Bt"] * (c["gamma"] + 1) * c["vocab"] * 4.0, "flops": L * flops}


# ------------------------------------------------------- results in 64 bits

def _labels(row, gamma):
    """tau and section (0 data, 1 mask, -1 padding) of the 2 gamma slots."""
    tau, sect = [0] * (2 * gamma), [-1] * (2 * gamma)
    for k, v in enumerate(row):
        if v > 0:
            tau[k] = tau[gamma + k] = v
            sect[k], sect[gamma + k] = 0, 1
        elif v == -1:
            tau[gamma + k], sect[gamma + k] = gamma + 1, 1
        elif v == -2:
            sect[k] = 0
    return tau, sect


def _visible(tau, sect):
    """Which new slot each slot sees: a data slot sees the data known no later
    than itself and the mask slots predicted later; a mask slot the data known
    before it and the mask slots predicted no earlier."""
    t = torch.tensor(tau, device="cuda")
    data = torch.tensor([s == 0 for s in sect], device="cuda")
    real = torch.tensor([s >= 0 for s in sect], device="cuda")
    before = torch.where(data[:, None], t[None, :] <= t[:, None], t[None, :] < t[:, None])
    return torch.where(data[None, :], before, ~before) & real[:, None] & real[None, :]


def _rotate(x, pos, theta):
    """Rotate-half RoPE of x [S][H][d] at pos [S], in 64 bits."""
    h = x.shape[-1] // 2
    f = theta ** (-torch.arange(h, dtype=torch.float64, device="cuda") / h)
    a = pos.double()[:, None, None] * f
    c, s = a.cos(), a.sin()
    return torch.cat([x[..., :h] * c - x[..., h:] * s, x[..., h:] * c + x[..., :h] * s], dim=-1)


def exact(case, seed):
    c = case
    if c["kind"] in ("accept", "sampled"):
        return None  # whole numbers
    si = _step_inputs(c, seed)
    w, L = si.w, si.q.shape[0]
    S, g, P = w.S, w.g, w.page_size
    n = si.prefix_len.tolist()
    maps = si.step_map.tolist()
    table = si.block_table.long()
    out = torch.zeros(si.q.shape, dtype=torch.float64, device="cuda")
    kept = [0] * w.Bt
    if c["kind"] == "step":
        hit = si.logits[:, : w.gamma].argmax(dim=-1) == si.draft
        kept = hit.long().cumprod(dim=1).sum(dim=1).tolist()
    # the caches after the commit (the rows of accepted drafts in 64 bits)
    written = []
    for b in range(w.Bt):
        tau, sect = _labels(maps[b], w.gamma)
        vis = _visible(tau, sect)
        pad = torch.tensor([s < 0 for s in sect], device="cuda")
        pos = n[b] + torch.arange(S, device="cuda") % w.gamma
        see = torch.cat([torch.ones(S, n[b], dtype=torch.bool, device="cuda"), vis], dim=1)
        pages = table[b, : (n[b] + P - 1) // P]
        for l in range(L):
            q, kn, vn = si.q[l, b].double(), si.k_new[l, b].double(), si.v_new[l, b].double()
            if c["rope"]:
                q, kn = _rotate(q, pos, _THETA), _rotate(kn, pos, _THETA)
            for h in range(w.Hkv):
                k = torch.cat([si.k_cache[l, pages, h].reshape(-1, w.d)[: n[b]].double(), kn[:, h]])
                v = torch.cat([si.v_cache[l, pages, h].reshape(-1, w.d)[: n[b]].double(), vn[:, h]])
                # padding slots may hold anything: they are seen by no row
                sc = torch.einsum("sgd,kd->sgk", q[:, h * g:(h + 1) * g], k) / math.sqrt(w.d)
                sc = sc.masked_fill(~see[:, None, :], float("-inf"))
                o = torch.einsum("sgk,kd->sgd", torch.softmax(sc, dim=-1), v)
                out[l, b, :, h * g:(h + 1) * g] = o.masked_fill(pad[:, None, None], 0.0)
            for r in range(kept[b]):
                slot, row = tau[: w.gamma].index(r + 1), n[b] + r
                written.append((l, int(table[b, row // P]), row % P, kn[slot], vn[slot]))
    if c["kind"] == "attention":
        return {"out": out[0]}
    kc, vc = si.k_cache.double(), si.v_cache.double()
    for l, page, row, kr, vr in written:
        kc[l, page, :, row] = kr
        vc[l, page, :, row] = vr
    return {"out": out, "accepted": None, "tokens": None, "argmax": None, "prefix_len": None, "k_cache": kc,
            "v_cache": vc}
