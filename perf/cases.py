"""The work that programs built on this package have it do, as measurable cases.

A next-scale generator calls the package once per scale: entropy maps of the scale's logits, keep
counts, selection, and then every layer on the kept tokens with the pruned ones restored from the
previous scale's residual cache. The kinds of case below are the ways in which it does so:

  scale       one scale through all layers, keep counts decided on the host (PrunedScaleRunner)
  graph       the same with every decision on the device, recorded once and replayed (DeviceScaleRunner)
  generation  all scales of a batch of images, from empty caches (MultiScaleRunner)
  layer       one layer of a text-conditioned backbone (rotary embedding, QK norm, cross-attention)
  head        selection of a scale straight from hidden states and the codebook head
  entropy     entropy maps and selection of several layers, from logits of either data type
  scores      the two other selection criteria (distance to the upsampled map, attention mass)

Sizes are those of the repository's configurations (the VAR-d16 256 and VAR-d30 512 shapes and the
width-2048 shape at 1024 and 2048) and generic ones around them.
"""
from __future__ import annotations

import math

import torch

import paper_2602_01345_b200 as nova
from paper_2602_01345_b200 import pipeline

DEV = "cuda:0"
V_CODEBOOK = 4096
EPS = 1e-6
SCALES_256 = (1, 2, 3, 4, 5, 6, 8, 10, 13, 16)

# Backbone shapes by width: heads (head size 64 up to 1920, 128 from 2048) and layers.
WIDTHS = {1024: (16, 16), 1280: (20, 20), 1536: (24, 24), 1920: (30, 30), 2048: (16, 32)}


def listed():
    return [
        # The smallest call sequence: one layer at the 16x16 scale for two images, five calls.
        {"name": "single_step_256", "kind": "scale", "layers": 1, "width": 1024, "heads": 16, "batch": 2, "h": 16, "w": 16,
         "prev": 13, "prior": 424, "keep": 0.5, "schedule": "forced", "fused": False, "modulated": False},
        # A whole class-conditional 256x256 generation: ten scales, the first ones tiny, nothing forced.
        {"name": "generation_256", "kind": "generation", "layers": 16, "width": 1024, "heads": 16, "batch": 8, "last": 16},
        # The last 512x512 scale with adaptive LayerNorm, head size 64, keep counts that differ by layer and image.
        {"name": "scale_512_adaln", "kind": "scale", "layers": 30, "width": 1920, "heads": 30, "batch": 4, "h": 32, "w": 32,
         "prev": 24, "prior": 1216, "keep": 0.5, "schedule": "paper", "fused": True, "modulated": True},
        # An early accelerated 1024x1024 scale for one image: few rows against 32 layers of weights.
        {"name": "scale_1024_early", "kind": "scale", "layers": 32, "width": 2048, "heads": 16, "batch": 1, "h": 20, "w": 20,
         "prev": 16, "prior": 521, "keep": 0.75, "schedule": "forced", "fused": True, "modulated": False},
        # A middle 1024x1024 scale before the trigger has fired: every token is kept.
        {"name": "scale_1024_dense", "kind": "scale", "layers": 32, "width": 2048, "heads": 16, "batch": 4, "h": 32, "w": 32,
         "prev": 24, "prior": 1497, "keep": 1.0, "schedule": "forced", "fused": True, "modulated": False},
        # The last 1024x1024 scale of one image in a serving loop: recorded once, replayed per image.
        {"name": "scale_1024_graph", "kind": "graph", "layers": 32, "width": 2048, "heads": 16, "batch": 1, "h": 64, "w": 64,
         "prev": 48, "prior": 6425, "keep": 0.25, "schedule": "forced", "fused": True, "modulated": False},
        # The repository's benchmark: the last 1024x1024 scale for four images, half of the tokens kept.
        {"name": "scale_1024_batch4", "kind": "scale", "layers": 32, "width": 2048, "heads": 16, "batch": 4, "h": 64, "w": 64,
         "prev": 48, "prior": 6425, "keep": 0.5, "schedule": "forced", "fused": True, "modulated": False},
        # The last 2048x2048 scale: 16384 tokens, a fifth kept, 27000 prior keys.
        {"name": "scale_2048", "kind": "scale", "layers": 32, "width": 2048, "heads": 16, "batch": 1, "h": 128, "w": 128,
         "prev": 96, "prior": 26137, "keep": 0.2, "schedule": "forced", "fused": True, "modulated": False},
        # A layer of a text-conditioned backbone on a 40x40 scale, prompts of different lengths.
        {"name": "layer_text_1024", "kind": "layer", "width": 2048, "heads": 16, "batch": 2, "h": 40, "w": 40, "prev": 32,
         "prior": 2521, "keep": 0.5, "cond": 128},
        # A decoder that has the hidden states at hand selects without ever writing the logits.
        {"name": "head_1024", "kind": "head", "width": 2048, "batch": 4, "n": 4096, "codes": 4096, "keep": 0.5},
        # Entropy and selection of eight layers from 32-bit logits.
        {"name": "entropy_f32", "kind": "entropy", "layers": 8, "batch": 4, "n": 1600, "codes": 4096, "dtype": "f32", "keep": 0.5},
        # The selection-criterion comparison at the 512x512 shape's last scale.
        {"name": "scores_512", "kind": "scores", "width": 1920, "heads": 30, "batch": 2, "h": 32, "w": 32, "prev": 24,
         "prior": 1216, "keep": 0.5},
    ]


# ---- drawn cases ---------------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scale(rng, kind):
    width = rng.choice(sorted(WIDTHS))
    heads, layers = WIDTHS[width]
    while True:
        h = _log_int(rng, 8, 96 if width == 2048 else 40)
        w = h if rng.random() < 0.7 else max(8, min(96, h + rng.randint(-h // 3, h // 3)))
        c = {"kind": kind, "layers": max(1, rng.randint(layers // 4, layers)), "width": width, "heads": heads,
             "batch": rng.choice((1, 1, 2, 3, 4, 5, 8)), "h": h, "w": w, "prev": max(1, int(h * rng.uniform(0.6, 0.85))),
             "prior": int(h * w * rng.uniform(1.0, 1.8)), "keep": round(rng.uniform(0.2, 1.0), 3),
             "schedule": rng.choice(("forced", "paper")), "fused": rng.random() < 0.6,
             "modulated": width < 2048 and rng.random() < 0.5}
        if c["batch"] * h * w <= 16384 and work(c)["flops"] <= (3.0e13 if width == 2048 else 1.5e13):
            return c


def draw(rng):
    kind = rng.choice(("scale", "scale", "scale", "graph", "generation", "layer", "head", "entropy", "scores"))
    if kind in ("scale", "graph"):
        return _draw_scale(rng, kind)
    width = rng.choice(sorted(WIDTHS))
    heads, layers = WIDTHS[width]
    if kind == "generation":
        return {"kind": kind, "layers": rng.randint(4, 16), "width": min(width, 1536), "heads": WIDTHS[min(width, 1536)][0],
                "batch": rng.randint(1, 8), "last": rng.randint(12, 24)}
    if kind == "layer":
        h = _log_int(rng, 12, 64)
        return {"kind": kind, "width": width, "heads": heads, "batch": rng.randint(1, 4), "h": h, "w": h, "prev": int(h * 0.8),
                "prior": int(h * h * rng.uniform(1.0, 1.8)), "keep": round(rng.uniform(0.2, 1.0), 3), "cond": rng.randint(16, 256)}
    if kind == "head":
        return {"kind": kind, "width": width, "batch": rng.randint(1, 4), "n": _log_int(rng, 100, 4096),
                "codes": rng.choice((1024, 2048, 4096)), "keep": round(rng.uniform(0.2, 0.8), 3)}
    if kind == "entropy":
        return {"kind": kind, "layers": rng.randint(1, 16), "batch": rng.randint(1, 4), "n": _log_int(rng, 64, 4096),
                "codes": rng.choice((1024, 2048, 4096)), "dtype": rng.choice(("f32", "bf16")),
                "keep": round(rng.uniform(0.2, 0.8), 3)}
    h = _log_int(rng, 10, 40)
    return {"kind": kind, "width": width, "heads": heads, "batch": rng.randint(1, 4), "h": h, "w": h, "prev": int(h * 0.8),
            "prior": int(h * h * rng.uniform(1.0, 1.5)), "keep": round(rng.uniform(0.2, 0.8), 3)}


# ---- inputs ----------------------------------------------------------------------------------------
class _Inputs:
    """Seeded random tensors on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed * 7919 + 17)

    def normal(self, shape, std=1.0, mean=0.0):
        x = torch.empty(shape, dtype=torch.bfloat16, device=DEV)
        return x.normal_(mean, std, generator=self.g)

    def uniform(self, shape, lo, hi):
        return torch.empty(shape, dtype=torch.float32, device=DEV).uniform_(lo, hi, generator=self.g)

    def weights(self, C, F):
        """One block: N(0, 0.02^2) as after initialisation, LayerNorm gains around 1."""
        shapes = {"ln1_g": (C,), "ln1_b": (C,), "w_qkv": (3 * C, C), "b_qkv": (3 * C,), "w_o": (C, C), "b_o": (C,),
                  "ln2_g": (C,), "ln2_b": (C,), "w_fc1": (F, C), "b_fc1": (F,), "w_fc2": (C, F), "b_fc2": (C,)}
        return {n: self.normal(s, 0.02, 1.0 if n in ("ln1_g", "ln2_g") else 0.0) for n, s in shapes.items()}

    def modulation(self, B, C):
        return {n: self.normal((B, C), 0.2, 1.0 if n.startswith("gate") else 0.0) for n in nova.binding.MODULATION_NAMES}

    def temperatures(self, B, h, w, lo, hi):
        """[B, h*w] inverse temperatures: a smooth field, half of it near lo and half near hi, so that the
        uncertain tokens lie together as they do in an image."""
        y = (torch.arange(h, device=DEV, dtype=torch.float32) + 0.5) / h
        x = (torch.arange(w, device=DEV, dtype=torch.float32) + 0.5) / w
        amp, fy, fx, ph = (self.uniform((B, 4, 1, 1), a, b) for a, b in ((0.5, 1.5), (0.3, 2.0), (0.3, 2.0), (0.0, 6.283)))
        f = (amp * torch.cos(6.2832 * (fy * y[None, None, :, None] + fx * x[None, None, None, :]) + ph)).sum(1).reshape(B, -1)
        f = (f - f.mean(1, keepdim=True)) / f.std(1, keepdim=True, correction=0).clamp_min(1e-6)
        return lo + (hi - lo) * torch.sigmoid(5.0 * f)

    def logits(self, a, V, dtype=torch.bfloat16):
        """[B, N] inverse temperatures -> [B, N, V] logits; a spread of the temperature itself keeps the
        entropies of neighbouring tokens apart."""
        z = torch.empty((*a.shape, V), dtype=dtype, device=DEV).normal_(generator=self.g)
        a = a * self.uniform(a.shape, 0.95, 1.05)
        return z.mul_(a.unsqueeze(-1).to(dtype))

    def layer_factors(self, L):
        return self.uniform((L,), 0.8, 1.25).tolist()

    def history(self, B, t):
        """Mean entropies of scales 1..t as a program has kept them: rising, a little different per image."""
        return (torch.linspace(2.0, 7.0, t).repeat(B, 1) + self.uniform((B, t), -0.1, 0.1).cpu()).contiguous()


def _scales_up_to(last):
    return SCALES_256 if last == 16 else tuple(sorted({max(1, round(last * s / 16)) for s in SCALES_256}))


def _schedule(c, t):
    if c["schedule"] == "paper":        # Eq. 11-13 at the scale where pruning begins: about half, by layer and image
        return nova.SchedParams(force_act_scale=t)
    return nova.SchedParams(force_act_scale=t, force_keep_ratio=c["keep"])


def _kv(r, L, B, rows, prior, C):
    """Caches of all layers, one allocation each, filled as far as the earlier scales did."""
    k, v = (torch.zeros((L, B, rows, C), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    for x in (k, v):
        for j in range(L):
            x[j, :, :prior] = r.normal((B, prior, C))
    return k, v, torch.full((L, B), prior, dtype=torch.int32, device=DEV)


def _selected(ctx, ent, keep):
    """Selection as a program that drives one layer by hand does it: returns the index lists."""
    B, N = ent.shape
    k = torch.full((B,), max(1, int(keep * N)), dtype=torch.int32)
    M = int(k.sum())
    keep_idx = torch.empty((M,), dtype=torch.int32, device=DEV)
    prune_idx = torch.empty((B * N - M,), dtype=torch.int32, device=DEV)
    cu = torch.empty((B + 1,), dtype=torch.int32, device=DEV)
    nova.nova_select_topk(ctx, ent, k, keep_idx, prune_idx, cu)
    return keep_idx, prune_idx, cu


def _prepare_scale(c, r, ctx):
    B, h, w, L, C = c["batch"], c["h"], c["w"], c["layers"], c["width"]
    t, F, rows = 10, 4 * C, c["prior"] + h * w
    weights = [r.weights(C, F) for _ in range(L)]
    k, v, kv_len = _kv(r, L, B, rows, c["prior"], C)
    prev = [r.normal((B, c["prev"], c["prev"], C)) for _ in range(L)]
    a = r.temperatures(B, h, w, 0.5, 6.0)
    logits = [r.logits(a * f, V_CODEBOOK) for f in r.layer_factors(L)]
    x_in = r.normal((B, h * w, C))
    mod = [r.modulation(B, C) for _ in range(L)] if c["modulated"] else None
    s = {"k": k, "v": v, "kv_len": kv_len, "kv_len0": kv_len.clone(), "x_in": x_in, "logits": logits, "t": t,
         "sched": _schedule(c, t), "hist": r.history(B, t), "keep_alive": weights}
    args = (ctx, weights, c["heads"], B, h, w, rows, list(k.unbind(0)), list(v.unbind(0)), list(kv_len.unbind(0)), prev)
    if c["kind"] == "scale":
        s["runner"] = pipeline.PrunedScaleRunner(*args, eps=EPS, modulation=mod, fused_restore=c["fused"])
    else:
        hist = s["hist"].t().contiguous().to(DEV)
        s["runner"] = pipeline.DeviceScaleRunner(*args, s["sched"], t, hist, V_CODEBOOK, eps=EPS, x_in=x_in,
                                                 layer_logits=logits, scale_entropy=False, modulation=mod,
                                                 fused_restore=c["fused"])
        s["runner"].capture()
    return s


def _prepare_generation(c, r, ctx):
    B, L, C = c["batch"], c["layers"], c["width"]
    scales = _scales_up_to(c["last"])
    T = len(scales)
    # mean entropy over the scales as a rising sigmoid: the trigger fires a few scales before the last
    H = 4.5 + 3.5 * torch.sigmoid((torch.arange(1, T + 1) - 3.5 - r.uniform((B, 1), -1.0, 1.0).cpu()) / 0.9)
    env = torch.sqrt(2.0 * (math.log(V_CODEBOOK) - H)).to(DEV)
    fac = r.layer_factors(L)
    inputs = []
    for t, side in enumerate(scales):
        a = env[:, t:t + 1] * r.temperatures(B, side, side, 0.7, 1.3)
        inputs.append((r.normal((B, side * side, C)), r.logits(a, V_CODEBOOK), [r.logits(a * f, V_CODEBOOK) for f in fac]))
    return {"weights": [r.weights(C, 4 * C) for _ in range(L)], "heads": c["heads"], "batch": B, "scales": scales,
            "inputs": inputs, "sched": nova.SchedParams()}


def _prepare_layer(c, r, ctx):
    B, h, w, C, heads = c["batch"], c["h"], c["w"], c["width"], c["heads"]
    N, dh, rows = h * w, C // heads, c["prior"] + h * w
    ent = r.uniform((B, N), 1.0, 8.0)
    keep_idx, prune_idx, cu = _selected(ctx, ent, c["keep"])
    M = keep_idx.numel()
    pos = torch.arange(N, device=DEV, dtype=torch.float32)
    freq = 10000.0 ** (-torch.arange(dh // 4, device=DEV, dtype=torch.float32) / (dh // 4))
    ang = torch.cat([(pos // w)[:, None] * freq, (pos % w)[:, None] * freq], 1)      # rows, then columns
    ext = {"rope_cos": ang.cos().contiguous(), "rope_sin": ang.sin().contiguous(),
           "qk_gain_q": r.normal((C,), 0.1, 3.0), "qk_gain_k": r.normal((C,), 0.1, 3.0),
           "lnc_g": r.normal((C,), 0.02, 1.0), "lnc_b": r.normal((C,), 0.02), "w_q2": r.normal((C, C), 0.02),
           "b_q2": r.normal((C,), 0.02), "w_o2": r.normal((C, C), 0.02), "b_o2": r.normal((C,), 0.02),
           "cond_k": r.normal((B, c["cond"], C)), "cond_v": r.normal((B, c["cond"], C)),
           "cond_len": (c["cond"] * r.uniform((B,), 0.3, 1.0)).to(torch.int32)}
    k, v, kv_len = _kv(r, 1, B, rows, c["prior"], C)
    shape = nova.BlockShape(B, N, C, heads, 4 * C, rows, M)
    ctx.ensure_workspace(shape)
    x = r.normal((B, N, C))
    return {"w": nova.BlockWeights(r.weights(C, 4 * C), EPS), "ext": ext, "shape": shape, "x": x, "keep_idx": keep_idx,
            "prune_idx": prune_idx, "cu": cu, "k": k[0], "v": v[0], "kv_len": kv_len[0], "kv_len0": kv_len[0].clone(),
            "prev": r.normal((B, c["prev"], c["prev"], C)), "h": h, "w_tokens": w, "y": torch.empty((M, C), dtype=torch.bfloat16, device=DEV),
            "x_out": torch.empty_like(x), "cache_out": torch.empty_like(x)}


def _prepare_head(c, r, ctx):
    B, N, C, V = c["batch"], c["n"], c["width"], c["codes"]
    # a head of this scale gives logits of the spread that the entropy maps are taken at
    amp = r.uniform((B, N, 1), 0.2, 3.0)
    return {"x": (r.normal((B, N, C)) * amp).to(torch.bfloat16), "head": r.normal((V, C), 1.0 / math.sqrt(C)), "bias": r.normal((V,), 0.1),
            "ent": torch.empty((B, N), device=DEV), "mean": torch.empty((B,), device=DEV), "keep": c["keep"]}


def _prepare_entropy(c, r, ctx):
    B, N, L = c["batch"], c["n"], c["layers"]
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    a = r.temperatures(B, 1, N, 0.5, 6.0)
    counts = (N * c["keep"] * r.uniform((L, B), 0.8, 1.2)).clamp(1, N).to(torch.int32)
    new = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)  # noqa: E731
    return {"logits": [r.logits(a * f, c["codes"], dt) for f in r.layer_factors(L)], "counts": counts,
            "ent": torch.empty((L, B, N), device=DEV), "mean": torch.empty((L, B), device=DEV), "keep_idx": new(L, B * N),
            "prune_idx": new(L, B * N), "cu": new(L, B + 1), "pos": new(L, B, N)}


def _prepare_scores(c, r, ctx):
    B, N, C = c["batch"], c["h"] * c["w"], c["width"]
    k, _, kv_len = _kv(r, 1, B, c["prior"] + N, c["prior"], C)
    return {"x": r.normal((B, N, C)), "prev": r.normal((B, c["prev"], c["prev"], C)), "h": c["h"], "w_tokens": c["w"],
            "q": r.normal((B, N, C)), "key": r.normal((B, N, C)), "k": k[0], "kv_len": kv_len[0], "heads": c["heads"],
            "keep": c["keep"], "mse": torch.empty((B, N), device=DEV), "mass": torch.empty((B, N), device=DEV)}


_PREPARE = {"scale": _prepare_scale, "graph": _prepare_scale, "generation": _prepare_generation, "layer": _prepare_layer,
            "head": _prepare_head, "entropy": _prepare_entropy, "scores": _prepare_scores}


def prepare(case, seed):
    ctx = nova.Context(0)
    s = _PREPARE[case["kind"]](case, _Inputs(seed), ctx)
    s["ctx"], s["kind"] = ctx, case["kind"]
    return s


# ---- one pass ----------------------------------------------------------------------------------------
def _run_scale(s):
    r = s["runner"]
    s["kv_len"].copy_(s["kv_len0"])        # every pass continues from the caches of the earlier scales
    x_out, _ = r.run_scale(s["x_in"], s["logits"], s["sched"], s["t"], s["hist"])
    return {"x_out": x_out, "cache_out": r.cache_out, "cu_keep": r.cu_keep, "ent": r.ent, "mean": r.mean, "k": s["k"], "v": s["v"],
            "kv_len": s["kv_len"]}


def _run_graph(s):
    r = s["runner"]
    s["kv_len"].copy_(s["kv_len0"])
    x_out = r.replay()
    return {"x_out": x_out, "cache_out": r.cache_out, "keep": r.keep, "cu_keep": r.cu_keep, "ent": r.ent, "mean": r.mean, "k": s["k"],
            "v": s["v"], "kv_len": s["kv_len"]}


def _run_generation(s):
    gen = pipeline.MultiScaleRunner(s["ctx"], s["weights"], s["heads"], s["batch"], s["scales"], eps=EPS)
    xs = []
    for t, (x_in, scale_logits, layer_logits) in enumerate(s["inputs"], 1):
        x_out, _, _ = gen.run_scale(t, x_in, scale_logits, layer_logits, s["sched"])
        xs.append(x_out)
    return {"x_out": xs, "history": gen.hbar_scale, "k": gen.k_caches, "v": gen.v_caches, "kv_len": gen.kv_len}


def _run_layer(s):
    ctx = s["ctx"]
    s["kv_len"].copy_(s["kv_len0"])
    nova.nova_pruned_block_forward_ext(ctx, s["w"], None, s["ext"], s["shape"], s["x"], s["keep_idx"], s["cu"], s["k"], s["v"],
                                       s["kv_len"], True, s["y"])
    nova.nova_restore_from_cache(ctx, s["x"], s["y"], s["keep_idx"], s["prune_idx"], s["cu"], s["prev"], s["h"], s["w_tokens"],
                                 s["x_out"], s["cache_out"])
    return {n: s[n] for n in ("y", "x_out", "cache_out", "k", "v", "kv_len")}


def _run_head(s):
    nova.nova_head_entropy(s["ctx"], s["x"], s["head"], s["bias"], s["ent"], s["mean"])
    return [s["ent"], s["mean"], *_selected(s["ctx"], s["ent"], s["keep"])]


def _run_entropy(s):
    nova.nova_scale_entropy_layers(s["ctx"], s["logits"], s["ent"], s["mean"])
    nova.nova_select_topk_grouped(s["ctx"], s["ent"], s["counts"], s["keep_idx"], s["prune_idx"], s["cu"], s["pos"])
    return {n: s[n] for n in ("ent", "mean", "keep_idx", "prune_idx", "cu", "pos")}


def _run_scores(s):
    nova.nova_score_mse(s["ctx"], s["x"], s["prev"], s["h"], s["w_tokens"], s["mse"])
    nova.nova_score_attention_mass(s["ctx"], s["q"], s["key"], s["k"], s["kv_len"], s["heads"], s["mass"])
    return [s["mse"], s["mass"], _selected(s["ctx"], s["mse"], s["keep"])]


_RUN = {"scale": _run_scale, "graph": _run_graph, "generation": _run_generation, "layer": _run_layer, "head": _run_head,
        "entropy": _run_entropy, "scores": _run_scores}


def run(state):
    return _RUN[state["kind"]](state)


# ---- what a pass cannot do without -----------------------------------------------------------------------
def _block_work(B, N, C, prior, kept):
    """One layer: its weights, prior K/V, new K/V, previous and new residual cache; GEMMs and attention.
    (What passes from layer to layer, x, is counted once per scale by the caller.)"""
    M, params = B * kept, 12 * C * C
    nbytes = 2 * params + 2 * 2 * C * (B * prior + M) + 2 * B * N * C
    return nbytes, 2.0 * M * params + 4.0 * B * kept * (prior + kept) * C


def work(case):
    c, kind = case, case["kind"]
    if kind in ("scale", "graph", "layer"):
        B, N, C, L = c["batch"], c["h"] * c["w"], c["width"], c.get("layers", 1)
        keep = 0.55 if c.get("schedule") == "paper" else c["keep"]
        kept = max(1, round(keep * N))
        nbytes, flops = _block_work(B, N, C, c["prior"], kept)
        if kept < N:
            nbytes += 2 * B * c["prev"] ** 2 * C
        if kind == "layer":
            nbytes += 2 * (2 * C * C + 2 * B * c["cond"] * C)
            flops += 4.0 * B * kept * C * C + 4.0 * B * kept * 0.65 * c["cond"] * C
        else:
            nbytes += B * N * (2 * V_CODEBOOK + 4)
        return {"bytes": L * nbytes + 4 * B * N * C, "flops": L * flops}
    if kind == "generation":
        B, C, L = c["batch"], c["width"], c["layers"]
        nbytes, flops, prior = 0.0, 0.0, 0
        for t, side in enumerate(_scales_up_to(c["last"]), 1):
            N = side * side
            kept = max(1, round(N * {8: 0.75, 9: 0.43, 10: 0.19}.get(t, 1.0)))     # what the schedule keeps of these inputs
            b, f = _block_work(B, N, C, prior, kept)
            nbytes += L * b + (L + 1) * 2 * B * N * V_CODEBOOK + 4 * B * N * C
            flops += L * f
            prior += kept
        return {"bytes": nbytes, "flops": flops}
    if kind == "head":
        rows = c["batch"] * c["n"]
        return {"bytes": 2 * c["width"] * (rows + c["codes"]) + 8 * rows, "flops": 2.0 * rows * c["width"] * c["codes"]}
    if kind == "entropy":
        rows = c["layers"] * c["batch"] * c["n"]
        return {"bytes": rows * (c["codes"] * (4 if c["dtype"] == "f32" else 2) + 12), "flops": 5.0 * rows * c["codes"]}
    B, N, C = c["batch"], c["h"] * c["w"], c["width"]
    return {"bytes": 2 * B * C * (3 * N + c["prev"] ** 2 + c["prior"]) + 16 * B * N, "flops": 2.0 * B * N * (N + c["prior"]) * C}


def tolerance(case):
    """Measured against a composition of library operations: with activations rounded to bf16 at the
    same places but every sum in another order, and with nothing rounded in between, outputs differ
    (2-norm) by 2e-3 to 4e-3 after one layer, 1.2e-2 after 16 and 1.2e-2 to 2e-2 after 30 to 32, single
    values by 0.05 after one layer and up to 0.33 after 32. Entropies and scores, sums of 32-bit terms,
    differ by up to 1e-6 from their 64-bit values; near-ties among them may change places."""
    c = case
    if c["kind"] in ("head", "entropy", "scores"):
        return {"rel": 5e-6, "max": 1e-4, "differ": 0.005}
    L = c.get("layers", 1)
    return {"rel": min(0.03, 0.01 * math.sqrt(L)), "max": min(0.9, 0.2 * math.sqrt(L))}
