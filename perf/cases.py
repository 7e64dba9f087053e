"""What a user of the framework has it do, as measurable cases.

Each case is one call (or the short sequence of calls that belongs together in
a sampling program) through the public entry points of the package: whole
generations, a refresh plus a reverse step of a model, blocks of backbone
layers in the three regimes of the sampling loop (whole canvas, block steps
over a KV context, causal prefill), and the building blocks (GEMM, attention,
output head, the two paper samplers).  Model sizes are the presets of
``workloads``; depths are cut to a few layers where one layer is what repeats.

``exact`` restates each case in plain torch, in 64 bits, from the same inputs.
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

import paper_2609_37924_gb300.tadm as T
import workloads as wl

# Model sizes by name: the presets' widths, with the vocabulary and the low-rank fusion width they use.
DIMS = {"tiny": wl.TINY, "small": wl.SMALL, "block": wl.BLOCK, "posttrain": wl.POSTTRAIN,
        "posttrain_g3": wl.POSTTRAIN_G3}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # A whole generation of the fp32 model (4 prompts, 32 + 96 tokens, 32 steps, a refresh every 4th), then the
        # logits of a held-out canvas: 300 small launches per step group, where latency counts.
        {"name": "tiny_generate_f32", "kind": "generate", "dims": "tiny", "batch": 4, "prompt": 32, "gen": 96,
         "steps": 32, "K": 4},
        # Unconditional generation, whole canvas of 1024 positions, batch 16: two layers of the anchor network, the
        # work that repeats in every step of the benchmark (attention of hd 64, 16384-row GEMMs).
        {"name": "small_layers_b16", "kind": "layers", "dims": "small", "batch": 16, "rows": 1024, "ctx": 0, "layers": 2},
        # The whole small model, one refresh and one reverse step that also returns its logits (scoring, or a
        # program's own sampler): 8 + 4 layers, gated-MLP fusion, output head.
        {"name": "small_step_logits", "kind": "step", "dims": "small", "batch": 4, "rows": 1024, "ctx": 0,
         "anchor": 8, "denoise": 4, "vocab": 32768, "logits": True},
        # One sequence, one 32-token block over a committed context: the latency case of block diffusion, bound by
        # reading the weights once (refresh, fusion, denoiser, head over 128000 tokens).
        {"name": "block_step_b1", "kind": "step", "dims": "block", "batch": 1, "rows": 32, "ctx": 1024,
         "anchor": 2, "denoise": 2, "vocab": 128000, "logits": False},
        # The serving batch of the block model: 32 sequences x 32 active rows over a 1024-token context.
        {"name": "block_layers_b32", "kind": "layers", "dims": "block", "batch": 32, "rows": 32, "ctx": 1024, "layers": 2},
        # The 27 B model's block step at its batch of 8 (256 rows, weight-streaming GEMMs), with the paired-attention
        # fusion; vocabulary cut so that the head has about the share it has at full depth.
        {"name": "posttrain_step_b8", "kind": "step", "dims": "posttrain", "batch": 8, "rows": 32, "ctx": 512,
         "anchor": 2, "denoise": 1, "vocab": 32768, "logits": False},
        # Prompt prefill (causal fresh pass, 8 prompts of 512 tokens) and the refresh of the first block after it.
        {"name": "block_prefill_b8", "kind": "prefill", "dims": "block", "batch": 8, "prompt": 512, "rows": 32,
         "layers": 2},
        # The fused output head on gathered rows (ragged count), 128000 tokens.
        {"name": "head_block_v128000", "kind": "head", "rows": 1500, "d": 2048, "vocab": 128000},
        # Attention of a block step of the 27 B model over a long context: GQA 32 / 16, hd 128.
        {"name": "attn_block_step_ctx2000", "kind": "attention", "batch": 8, "heads": 32, "kv_heads": 16, "hd": 128,
         "rows": 32, "ctx": 2000, "causal": False, "window": 0},
        # The plain GEMM building block at a ragged size.
        {"name": "gemm_ragged", "kind": "gemm", "m": 1111, "n": 3000, "k": 2056, "out": "f32"},
        # One step of the entropy-bound sampler on the post-training canvas (8 x 256 positions, 262144 tokens), with
        # the probabilities that self-conditioning reads.
        {"name": "eb_update_v262144", "kind": "eb", "batch": 8, "rows": 512, "first": 256, "vocab": 262144, "probs": "bf16"},
        # One ReMDM step on the small workload's canvas: remasks, and nucleus draws for one masked position in eight.
        {"name": "remdm_update_v32768", "kind": "remdm", "batch": 16, "rows": 1024, "first": 256, "vocab": 32768,
         "p_unmask": 0.125},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate", "layers", "layers", "layers", "step", "step", "step", "prefill", "head", "attention",
                       "attention", "gemm", "eb", "remdm"])
    if kind == "generate":
        gen, steps = rng.randint(32, 96), rng.randint(8, 32)
        return {"kind": kind, "dims": "tiny", "batch": rng.randint(3, 4), "prompt": rng.randint(7, 32), "gen": gen,
                "steps": steps, "K": rng.choice([1, 2, 4, 8])}
    if kind == "layers":
        dims = rng.choice(["tiny", "small", "small", "block", "block", "posttrain", "posttrain_g3"])
        if dims in ("tiny", "small"):                  # whole canvases
            rows = _log(rng, 40, 1024)
            batch = _log(rng, 1, 16 if dims == "small" else 4)
            return {"kind": kind, "dims": dims, "batch": batch, "rows": rows, "ctx": 0, "layers": 2}
        batch = _log(rng, 1, 32 if dims == "block" else 8)
        return {"kind": kind, "dims": dims, "batch": batch, "rows": rng.choice([16, 24, 32, 32, 32]),
                "ctx": _log(rng, 64, 1024 if dims == "block" else 512), "layers": 2}
    if kind == "step":
        dims = rng.choice(["small", "block", "block", "posttrain", "posttrain_g3"])
        if dims == "small":
            return {"kind": kind, "dims": dims, "batch": _log(rng, 1, 4), "rows": _log(rng, 100, 1024), "ctx": 0,
                    "anchor": rng.randint(2, 8), "denoise": rng.randint(1, 4), "vocab": rng.choice([32768, 30522]),
                    "logits": rng.random() < 0.5}
        return {"kind": kind, "dims": dims, "batch": _log(rng, 1, 8), "rows": rng.choice([16, 32, 32]),
                "ctx": _log(rng, 64, 1024 if dims == "block" else 512), "anchor": rng.randint(1, 2), "denoise": 1,
                "vocab": rng.choice([32768, 50257]) if dims != "block" else 128000, "logits": False}
    if kind == "prefill":
        return {"kind": kind, "dims": "block", "batch": _log(rng, 1, 8), "prompt": _log(rng, 33, 512),
                "rows": rng.choice([16, 32]), "layers": rng.randint(1, 2)}
    if kind == "head":
        d = rng.choice([768, 2048, 2048, 5376])
        return {"kind": kind, "rows": _log(rng, 8, 1500 if d < 5000 else 256), "d": d,
                "vocab": rng.choice([32768, 50257, 128000])}
    if kind == "attention":
        if rng.random() < 0.5:                          # whole canvases, hd 64
            rows = _log(rng, 60, 1024)
            return {"kind": kind, "batch": _log(rng, 1, 16), "heads": 12, "kv_heads": 12, "hd": 64, "rows": rows, "ctx": 0,
                    "causal": rng.random() < 0.25, "window": 0}
        heads, kv = rng.choice([(16, 8), (32, 16)])
        return {"kind": kind, "batch": _log(rng, 1, 8), "heads": heads, "kv_heads": kv, "hd": 128,
                "rows": rng.choice([16, 31, 32, 64]), "ctx": _log(rng, 64, 2000), "causal": False,
                "window": rng.choice([0, 0, 1024])}
    if kind == "gemm":
        return {"kind": kind, "m": _log(rng, 16, 1111), "n": _log(rng, 64, 3000), "k": 8 * _log(rng, 16, 257),
                "out": rng.choice(["f32", "bf16"])}
    if kind == "eb":
        G, first = _log(rng, 32, 256), rng.randint(0, 256)
        return {"kind": kind, "batch": _log(rng, 1, 8), "rows": first + G, "first": first,
                "vocab": rng.choice([32768, 50257, 128000, 262144]), "probs": rng.choice(["none", "bf16", "f32"])}
    first = rng.randint(0, 256)
    return {"kind": kind, "batch": _log(rng, 1, 16), "rows": first + _log(rng, 64, 768), "first": first,
            "vocab": rng.choice([32768, 30522, 50257]), "p_unmask": rng.choice([0.03125, 0.125])}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _model(case):
    m = DIMS[case["dims"]]
    kind = case["kind"]
    if kind == "layers" or kind == "prefill":
        # the anchor latent is the output: no fusion, no denoiser; a small vocabulary, which nothing reads but the embedding
        return replace(m, n_shared=0, n_anchor=case["layers"], n_denoise=0, fusion="none", vocab=4096)
    if kind == "step":
        return replace(m, n_shared=0, n_anchor=case["anchor"], n_denoise=case["denoise"], vocab=case["vocab"])
    return m


def _weights(m, g):
    dt = torch.bfloat16 if m.dtype == "bf16" else torch.float32
    out = {}
    for s in wl.weight_specs(m):
        w = torch.randn(s.shape, generator=g, device="cuda", dtype=torch.float32 if s.kind != "matrix" else dt)
        out[s.name] = (w.mul_(0.02) if s.kind == "matrix" else w.mul_(0.05).add_(1.0 if s.kind == "gain" else 0.0)).to(dt)
    return out


def _canvas(m, g, batch, rows, masked):
    """Token ids with the given share of MASK."""
    z = torch.randint(0, m.vocab - 1, (batch, rows), generator=g, device="cuda", dtype=torch.int32)
    z[torch.rand((batch, rows), generator=g, device="cuda") < masked] = m.mask_id
    return z


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    g = _gen(seed)
    kind = case["kind"]
    r = {}
    if kind in ("generate", "layers", "step", "prefill"):
        m = _model(case)
        r["m"], r["w"] = m, _weights(m, g)
        B = case["batch"]
        if kind == "generate":
            r["prompt"] = _canvas(m, g, B, case["prompt"], 0.0)
            r["x"] = _canvas(m, g, B, case["prompt"] + case["gen"], 0.5)
            return r
        if case.get("ctx") or kind == "prefill":
            r["prompt"] = _canvas(m, g, B, case["ctx"] if kind != "prefill" else case["prompt"], 0.0)
        r["x"] = _canvas(m, g, B, case["rows"], 0.75)
        if kind == "step":     # the canvas of a later step: about half of the masks have become tokens
            later = _canvas(m, g, B, case["rows"], 0.5)
            r["x2"] = torch.where(r["x"] == m.mask_id, later, r["x"])
        return r
    if kind == "head":
        r["x"] = torch.randn((case["rows"], case["d"]), generator=g, device="cuda").to(torch.bfloat16)
        r["w"] = torch.randn((case["vocab"], case["d"]), generator=g, device="cuda", dtype=torch.bfloat16).mul_(0.05)
    elif kind == "attention":
        B, hd, kv = case["batch"], case["hd"], case["kv_heads"]
        n = case["ctx"] + case["rows"]
        stride = (n + 7) // 8 * 8
        rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
        r["q"] = rnd(B, case["heads"], case["rows"], hd)
        r["k"], r["v"] = rnd(B, kv, stride, hd), rnd(B, kv, hd, stride)
        r["n"] = n
    elif kind == "gemm":
        r["a"] = torch.randn((case["m"], case["k"]), generator=g, device="cuda").to(torch.bfloat16)
        r["b"] = torch.randn((case["n"], case["k"]), generator=g, device="cuda").to(torch.bfloat16)
    elif kind in ("eb", "remdm"):
        B, R, V = case["batch"], case["rows"], case["vocab"]
        rows = B * (R - case["first"]) if kind == "eb" else B * R
        # some positions are nearly decided, some open, some nearly flat
        scale = torch.tensor([3.0, 1.0, 2.0], device="cuda")[torch.randint(0, 3, (rows, 1), generator=g, device="cuda")]
        r["logits"] = torch.randn((rows, V), generator=g, device="cuda").mul_(scale)
        peak = torch.randint(0, V - 1, (rows, 1), generator=g, device="cuda")
        sure = torch.rand((rows, 1), generator=g, device="cuda") < 0.3
        r["logits"].scatter_add_(1, peak, torch.where(sure, 40.0, 4.0))
        z = torch.randint(0, V - 1, (B, R), generator=g, device="cuda", dtype=torch.int32)
        if kind == "remdm":
            gen = torch.arange(R, device="cuda") >= case["first"]
            z[(torch.rand((B, R), generator=g, device="cuda") < 0.6) & gen] = V - 1
        r["z"] = z
        r["seed"] = seed & 0xFFFFFFFF
    return r


def prepare(case, seed):
    s = {"case": case, **_inputs(case, seed)}
    kind = case["kind"]
    dev = dict(device="cuda")
    if kind in ("generate", "layers", "step", "prefill"):
        m, B = s["m"], case["batch"]
        if kind == "generate":
            total = case["prompt"] + case["gen"]
            s["tm"] = T.TadmModel(m, s["w"], max_batch=B, max_rows=total)
            s["out"] = torch.empty((B, total), dtype=torch.int32, **dev)
            s["cache"] = s["tm"].new_cache(B, total)
            s["logits"] = torch.empty((B * total, m.vocab), dtype=torch.float32, **dev)
            s["xt"] = s["x"].clone()
            return s
        R, P = case["rows"], s["prompt"].shape[1] if "prompt" in s else 0
        s["tm"] = T.TadmModel(m, s["w"], max_batch=B, max_rows=max(R, P), max_ctx=P + R if P else 0)
        s["cache"] = s["tm"].new_cache(B, R)
        s["h"] = s["cache"][:B * R * m.d_model * 4].view(torch.float32).view(B * R, m.d_model)
        if kind == "step":
            s["xt"] = s["x2"].clone()
            s["conf"] = torch.empty(B * R, dtype=torch.float32, **dev)
            s["fused"] = torch.empty((B * R, m.d_model), dtype=torch.float32, **dev)
            s["logits"] = torch.empty((B * R, m.vocab), dtype=torch.float32, **dev) if case["logits"] else None
        s["tm"].tadm_reset(B)
        if kind != "prefill" and P:
            s["tm"].tadm_prefill(s["prompt"])      # the committed context that the block's steps attend to
    elif kind == "head":
        s["scratch"] = torch.empty(T.tadm_head_scratch_size(case["rows"], case["vocab"], 1), dtype=torch.uint8, **dev)
        s["conf"] = torch.empty(case["rows"], dtype=torch.float32, **dev)
        s["tok"] = torch.empty(case["rows"], dtype=torch.int32, **dev)
    elif kind == "attention":
        s["o"] = torch.empty((case["batch"] * case["rows"], case["heads"] * case["hd"]), dtype=torch.bfloat16, **dev)
    elif kind == "gemm":
        s["c"] = torch.empty((case["m"], case["n"]), dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16, **dev)
    elif kind == "eb":
        n = s["logits"].shape[0]
        s["ent"] = torch.empty(n, dtype=torch.float32, **dev)
        s["zsum"] = torch.empty(n, dtype=torch.float32, **dev)
        dt = {"bf16": torch.bfloat16, "f32": torch.float32}.get(case["probs"])
        s["probs"] = torch.empty(s["logits"].shape, dtype=dt, **dev) if dt else None
    else:
        s["zt"] = s["z"].clone()
        s["action"] = torch.empty(s["logits"].shape[0], dtype=torch.int32, **dev)
    return s


# ------------------------------------------------------------------ one pass
STEPS = 16   # reverse steps of a block, of which the step cases run one


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "generate":
        tm = s["tm"]
        tm.tadm_generate(s["prompt"], s["out"], case["gen"], case["steps"], case["K"])
        tm.tadm_anchor_forward(s["x"], case["steps"], s["cache"])
        tm.tadm_denoise_step(s["xt"], case["steps"], case["steps"], 0, s["cache"], logits=s["logits"])
        return s["out"], s["logits"]
    if kind == "layers":
        s["tm"].tadm_anchor_forward(s["x"], STEPS, s["cache"])
        return s["h"]
    if kind == "prefill":
        s["tm"].tadm_reset(case["batch"])
        s["tm"].tadm_prefill(s["prompt"])
        s["tm"].tadm_anchor_forward(s["x"], STEPS, s["cache"])
        return s["h"]
    if kind == "step":
        s["tm"].tadm_anchor_forward(s["x"], STEPS, s["cache"])
        s["xt"].copy_(s["x2"])
        s["tm"].tadm_denoise_step(s["xt"], STEPS - 1, STEPS, case["rows"] // 2, s["cache"], logits=s["logits"],
                                  conf=s["conf"], fused=s["fused"])
        out = [s["h"], s["fused"], s["conf"], s["xt"]]
        return out + [s["logits"]] if case["logits"] else out
    V = case.get("vocab", 0)
    if kind == "head":
        T.tadm_head_confidence(s["x"], s["w"], V - 1, s["conf"], s["tok"], s["scratch"], 1)
        return s["conf"], s["tok"]
    if kind == "attention":
        T.tadm_attention(s["q"], s["k"], s["v"], s["o"], case["heads"], case["kv_heads"], case["rows"], case["ctx"],
                         case["causal"], 1, window=case["window"])
        return s["o"]
    if kind == "gemm":
        T.tadm_gemm(s["a"], s["b"], s["c"], 1)
        return s["c"]
    if kind == "eb":
        T.tadm_eb_update(s["z"], s["logits"], case["first"], V - 1, 0.6, 0.1, False, s["seed"], 3, s["ent"], s["probs"],
                         s["zsum"])
        out = [s["z"], s["ent"], s["zsum"]]
        return out + [s["probs"]] if s["probs"] is not None else out
    s["zt"].copy_(s["z"])
    T.tadm_remdm_update(s["zt"], s["logits"], case["first"], V - 1, 0.04, case["p_unmask"], 0.9, s["seed"], 5, s["action"])
    return s["zt"], s["action"]


# ------------------------------------------------------------------ what a pass cannot do without
def _layer_flops(m, M, keys, qkv=True):
    q, kv = m.n_heads * m.head_dim, m.n_kv_heads * m.head_dim
    proj = m.d_model * (q + 2 * kv) + q * m.d_model + 3 * m.d_model * m.ffn
    return 2.0 * M * proj + 4.0 * M * q * keys


def _params(m, layers):
    q, kv = m.n_heads * m.head_dim, m.n_kv_heads * m.head_dim
    return layers * (m.d_model * (q + 2 * kv) + q * m.d_model + 3 * m.d_model * m.ffn)


def work(case):
    kind = case["kind"]
    if kind in ("generate", "layers", "step", "prefill"):
        m = _model(case)
        es = 2 if m.dtype == "bf16" else 4
        B, d = case["batch"], m.d_model
        kv_bytes = lambda ctx, layers: 2.0 * B * m.n_kv_heads * m.head_dim * ctx * es * layers  # noqa: E731
        if kind == "layers":
            R, L = case["rows"], case["layers"]
            return {"bytes": es * _params(m, L) + kv_bytes(case["ctx"], L) + 4.0 * B * R * d + 4.0 * B * R,
                    "flops": L * _layer_flops(m, B * R, case["ctx"] + R)}
        if kind == "prefill":
            P, R, L = case["prompt"], case["rows"], case["layers"]
            return {"bytes": es * _params(m, L) + kv_bytes(P, L) + 4.0 * B * R * d,
                    "flops": L * (_layer_flops(m, B * P, (P + 1) / 2) + _layer_flops(m, B * R, P + R))}
        if m.fusion == "gated_mlp":
            fus = 14.0 * d * d                    # 2d x 5d and 4d x d
        else:
            r = m.fusion_rank
            fus = 3.0 * d * r + 16.0 * r * r
        head = float(m.vocab) * d
        if kind == "step":
            R, L = case["rows"], case["anchor"] + case["denoise"]
            outs = 4.0 * B * R * (2 * d + 2) + (4.0 * B * R * m.vocab if case["logits"] else 0.0)
            return {"bytes": es * (_params(m, L) + fus + head) + kv_bytes(case["ctx"], L) + outs,
                    "flops": L * _layer_flops(m, B * R, case["ctx"] + R) + 2.0 * B * R * (fus + head)}
        R, n = case["prompt"] + case["gen"], case["steps"]
        A = -(-n // case["K"])
        L = (n + 1) * m.n_denoise + (A + 1) * m.n_anchor
        heads = B * sum(case["gen"] - i * case["gen"] // n for i in range(n)) + B * R
        return {"bytes": es * _params(m, L) + es * (n + 1) * (fus + head) + 4.0 * B * R * m.vocab,
                "flops": L * _layer_flops(m, B * R, R) + 2.0 * B * R * (n + 1) * fus + 2.0 * heads * head}
    if kind == "head":
        return {"bytes": 2.0 * (case["rows"] + case["vocab"]) * case["d"] + 8.0 * case["rows"],
                "flops": 2.0 * case["rows"] * case["vocab"] * case["d"]}
    if kind == "attention":
        n, q = case["ctx"] + case["rows"], case["heads"] * case["hd"]
        keys = case["ctx"] + (case["rows"] + 1) / 2 if case["causal"] else n
        if case["window"]:
            keys = min(keys, case["window"] + case["rows"])
        return {"bytes": 2.0 * case["batch"] * (2 * case["rows"] * q + 2 * case["kv_heads"] * case["hd"] * min(n, keys + 1)),
                "flops": 4.0 * case["batch"] * case["rows"] * q * keys}
    if kind == "gemm":
        return {"bytes": 2.0 * (case["m"] + case["n"]) * case["k"] + (4.0 if case["out"] == "f32" else 2.0) * case["m"] * case["n"],
                "flops": 2.0 * case["m"] * case["n"] * case["k"]}
    B, R, V = case["batch"], case["rows"], case["vocab"]
    if kind == "eb":
        n = B * (R - case["first"])
        return {"bytes": n * V * (4.0 + {"none": 0, "bf16": 2, "f32": 4}[case["probs"]]) + 12.0 * n, "flops": 4.0 * n * V}
    n = B * (R - case["first"]) * 0.6 * case["p_unmask"]       # the rows that draw a token
    return {"bytes": 4.0 * n * V + 8.0 * B * R, "flops": 4.0 * n * V}


# ------------------------------------------------------------------ tolerances
def tolerance(case):
    kind = case["kind"]
    if kind == "generate":
        # fp32 throughout; a confidence tie that another order of sums breaks moves a token of one sequence
        return {"rel": 2e-5, "max": 1e-3, "differ": 0.01}
    if kind in ("layers", "step", "prefill"):
        if DIMS[case["dims"]].dtype == "f32":
            return {"rel": 2e-5, "max": 1e-3, "differ": 0.01}
        # bf16 operands, re-rounded in every layer
        return {"rel": 0.02, "max": 0.5, "differ": 0.01}
    if kind == "head":      # fp32 logits of 2048 to 5376 terms, exponentiated
        return {"rel": 5e-5, "max": 1e-3, "differ": 1e-3}
    if kind == "attention":
        return {"rel": 4e-3, "max": 0.1}
    if kind == "gemm":
        return {"rel": 1e-5, "max": 1e-4} if case["out"] == "f32" else {"rel": 1e-3, "max": 0.02}
    if kind == "eb":        # fp32 sums; probabilities rounded to bf16 may move by one unit in the last place
        return {"rel": 2e-4, "max": 0.01, "differ": 5e-3}
    return {"differ": 1e-3}  # a draw on the edge of a fp32 cumulative sum


# ------------------------------------------------------------------ the same in 64 bits
F64 = torch.float64


def _mm(x, w, rows=16384):
    """x W^T in fp64, a slab of W's rows at a time."""
    return torch.cat([x @ w[i:i + rows].to(F64).T for i in range(0, w.shape[0], rows)], 1)


def _rms(x, gain, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain.to(F64)


def _ln(x, w, b, eps):
    return (x - x.mean(-1, keepdim=True)) * torch.rsqrt(x.var(-1, unbiased=False, keepdim=True) + eps) * w.to(F64) + b.to(F64)


def _attend(q, k, v, scale, see):
    """softmax(q k^T scale) v with the visible keys `see` [rows, keys]; heads of a group share k, v."""
    out = torch.empty_like(q)
    rep = q.shape[1] // k.shape[1]
    for b in range(q.shape[0]):
        kb, vb = k[b].repeat_interleave(rep, 0), v[b].repeat_interleave(rep, 0)
        a = (q[b] @ kb.transpose(1, 2) * scale).masked_fill(~see, -math.inf)
        out[b] = torch.softmax(a, -1) @ vb
    return out


def _rope(x, pos, theta):
    half = x.shape[-1] // 2
    ang = pos.to(F64)[:, None] * theta ** (-torch.arange(half, device=x.device, dtype=F64) / half)
    c, s = ang.cos(), ang.sin()
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _see(rows, ctx, causal, window, device):
    p = ctx + torch.arange(rows, device=device)[:, None]
    j = torch.arange(ctx + rows, device=device)[None, :]
    see = torch.ones((rows, ctx + rows), dtype=torch.bool, device=device)
    if causal:
        see &= j <= p
    if window:
        see &= p - j < window
    return see


class _Ref:
    """The network in fp64: every layer keeps the keys and values of its committed context."""

    def __init__(self, m, w):
        self.m, self.w = m, w
        self.kv = {}
        self.ctx = 0

    def layer(self, net, i, index, x, B, causal, keep):
        m, w, p = self.m, self.w, "%s.%d." % (net, i)
        M, hd, hq, hk = x.shape[0], m.head_dim, m.n_heads, m.n_kv_heads
        R = M // B
        everywhere = m.global_every == 0 or (index + 1) % m.global_every == 0
        theta = m.rope_theta_global if everywhere and m.rope_theta_global > 0 else m.rope_theta
        y = _mm(_rms(x, w[p + "attn_norm"], m.norm_eps), w[p + "wqkv"])
        y = y.view(B, R, hq + 2 * hk, hd).transpose(1, 2)
        q, k, v = y[:, :hq], y[:, hq:hq + hk], y[:, hq + hk:]
        if m.qk_norm:
            q, k = _rms(q, w[p + "q_norm"], m.norm_eps), _rms(k, w[p + "k_norm"], m.norm_eps)
        pos = self.ctx + torch.arange(R, device=x.device)
        q, k = _rope(q, pos, theta), _rope(k, pos, theta)
        if index in self.kv:
            k, v = torch.cat([self.kv[index][0], k], 2), torch.cat([self.kv[index][1], v], 2)
        if keep:
            self.kv[index] = (k, v)
        o = _attend(q, k, v, 1.0 / math.sqrt(hd), _see(R, self.ctx, causal, 0 if everywhere else m.sliding_window, x.device))
        o = _mm(o.transpose(1, 2).reshape(M, hq * hd), w[p + "wo"])
        x = x + (_rms(o, w[p + "post_attn_norm"], m.norm_eps) if m.sandwich_norm else o)
        n = _rms(x, w[p + "ffn_norm"], m.norm_eps)
        gate, up = _mm(n, w[p + "wgu"][:m.ffn]), _mm(n, w[p + "wgu"][m.ffn:])
        act = torch.nn.functional.gelu(gate, approximate="tanh") if m.glu == "geglu" else torch.nn.functional.silu(gate)
        f = _mm(act * up, w[p + "wdown"])
        return x + (_rms(f, w[p + "post_ffn_norm"], m.norm_eps) if m.sandwich_norm else f)

    def stack(self, net, n, first, x, B, causal=False, keep=False):
        for i in range(n):
            x = self.layer(net, i, first + i, x, B, causal, keep)
        return x

    def embed(self, z):
        return self.w["embed"][z.reshape(-1).long()].to(F64)

    def anchor(self, z, causal=False, keep=False):
        return self.stack("anchor", self.m.n_anchor, 0, self.embed(z), z.shape[0], causal, keep)

    def prefill(self, z):
        h = self.anchor(z, True, True)
        # a fresh anchor: the paired-attention fusion is the identity there
        x = h if self.m.fusion != "gated_mlp" else self.fuse(z, z, h)
        self.stack("denoise", self.m.n_denoise, self.m.n_anchor, x, z.shape[0], True, True)
        self.ctx += z.shape[1]

    def fuse(self, z, z0, h):
        """h~ = Phi(c, cache): z the current canvas, z0 the refresh's, h its latent."""
        m, w, B = self.m, self.w, z.shape[0]
        c = self.embed(z)
        if m.fusion == "gated_mlp":
            u = torch.cat([_ln(c, w["fusion.ln_c.w"], w["fusion.ln_c.b"], m.norm_eps),
                           _ln(h, w["fusion.ln_h.w"], w["fusion.ln_h.b"], m.norm_eps)], 1)
            y = _mm(u, w["fusion.w_g1"]) + w["fusion.b_g1"].to(F64)
            g, a = torch.sigmoid(y[:, :m.d_model]), torch.nn.functional.gelu(y[:, m.d_model:])
            pre = h + g * (_mm(a, w["fusion.w2"]) + w["fusion.b2"].to(F64))
            return _ln(pre, w["fusion.ln_out.w"], w["fusion.ln_out.b"], m.norm_eps)
        c0 = self.embed(z0)
        r, fh = m.fusion_rank, m.fusion_heads
        scale = lambda t: torch.sqrt(t.square().mean(-1, keepdim=True) + 1e-6)  # noqa: E731
        sc, sh = scale(c0), scale(h)
        Z, Z0, U = _mm(c / sc, w["fusion.wc"]), _mm(c0 / sc, w["fusion.wc"]), _mm(h / sh, w["fusion.wh"])

        def mix(Zi):
            y = _mm(torch.cat([Zi, U], 1), w["fusion.wqkv"]).view(B, -1, 3 * fh, r // fh).transpose(1, 2)
            R = y.shape[2]
            o = _attend(y[:, :fh], y[:, fh:2 * fh], y[:, 2 * fh:], 1.0 / math.sqrt(r // fh), _see(R, 0, False, 0, y.device))
            Rr = Zi + _mm(o.transpose(1, 2).reshape(-1, r), w["fusion.wo"])
            return Rr + _mm(torch.nn.functional.silu(_mm(Rr, w["fusion.w1"])), w["fusion.w2"])

        M = mix(Z) - mix(Z0)
        F = torch.cat([U, Z0, Z - Z0, M], 1)
        gate = torch.sigmoid(_mm(torch.nn.functional.silu(_mm(F, w["fusion.wg1"])), w["fusion.wg2"]) + w["fusion.bg"].to(F64))
        return h + gate * sh * _mm(M, w["fusion.wup"])

    def logits(self, x, B):
        m, w = self.m, self.w
        x = self.stack("denoise", m.n_denoise, m.n_anchor, x, B)
        return _mm(_rms(x, w["final_norm"], m.norm_eps), w["embed"] if m.tied_lm_head else w["lm_head"])


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    kind = case["kind"]
    if kind == "remdm":      # whole numbers only
        return None
    r = _inputs(case, seed)
    if kind in ("generate", "layers", "step", "prefill"):
        m = r["m"]
        ref, B = _Ref(m, r["w"]), case["batch"]
        if "prompt" in r and kind != "generate":
            ref.prefill(r["prompt"])
        h = ref.anchor(r["x"])
        if kind == "generate":
            return None, ref.logits(ref.fuse(r["x"], r["x"], h), B)
        if kind != "step":
            return h
        fused = ref.fuse(r["x2"], r["x"], h)
        logits = ref.logits(fused, B)
        conf = torch.softmax(logits[:, :-1], 1).amax(1)          # MASK, the last id, is never predicted
        return [h, fused, conf, None, logits] if case["logits"] else [h, fused, conf, None]
    if kind == "head":
        logits = _mm(r["x"].to(F64), r["w"][:-1])
        return torch.softmax(logits, 1).amax(1), None
    if kind == "attention":
        q, k = r["q"].to(F64), r["k"][:, :, :r["n"]].to(F64)
        v = r["v"][..., :r["n"]].to(F64).transpose(2, 3)
        o = _attend(q, k, v, 1.0 / math.sqrt(case["hd"]),
                    _see(case["rows"], case["ctx"], case["causal"], case["window"], q.device))
        return o.transpose(1, 2).reshape(case["batch"] * case["rows"], -1)
    if kind == "gemm":
        return _mm(r["a"].to(F64), r["b"])
    ent, zsum, probs = [], [], []
    for i in range(0, r["logits"].shape[0], 256):
        l64 = r["logits"][i:i + 256].to(F64)
        l64[:, -1] = -math.inf
        a = (l64 - l64.amax(1, keepdim=True)) / 0.6
        q = a.exp()
        Z = q.sum(1)
        ent.append(Z.log() - (q * a.masked_fill(q == 0, 0.0)).sum(1) / Z)
        zsum.append(Z)
        if case["probs"] != "none":
            probs.append(q)
    out = [None, torch.cat(ent), torch.cat(zsum)]
    return out + [torch.cat(probs)] if probs else out
