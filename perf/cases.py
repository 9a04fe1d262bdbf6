"""Timed cases of the attention path: what a video-DiT denoising loop calls, from the smallest call to the largest.

A case is one problem (batch, heads, head_dim, latent grid, budgets and options) and the way it is called:
  call    da2_prepare + da2_attention_fwd on tensors that live on the GPU (the ordinary layer call)
  cached  da2_prepare_cached_scales + da2_attention_fwd: a later denoising step under the scales of the step before
  reuse   da2_refresh_operands + da2_attention_fwd: a later step under the block selection of the step before
  host    HostPipeline: pinned host tensors in and out
  map     da2_draft_map_noalloc: the low-resolution draft map alone, from region descriptors
Plans, workspaces, output buffers and pipelines are made in prepare(), as a denoising loop makes them once.
"""
import math

import torch
import torch.nn.functional as F

import paper_2609_32628_b200 as da2

_DEFAULTS = dict(mode="call", B=1, H=1, d=128, T=1, Hg=8, Wg=8, f16=0.0, f8=0.0, f4=0.0, head_scope=False,
                 balanced=False, prefix=0, k_outliers=False)


def _case(**kw):
    return {**_DEFAULTS, **kw}


def listed():
    return [
        # the smallest call: two heads of a 1,024-token latent; launches and host time are what it consists of
        _case(name="tiny", H=2, d=64, T=4, Hg=16, Wg=16, f8=0.25, f4=0.25),
        # a short preview clip on a ragged grid with all three formats at head_dim 64, two prompts in one batch
        _case(name="ragged_three_tier_d64", B=2, H=4, d=64, T=7, Hg=27, Wg=43, f16=0.15, f8=0.25, f4=0.30),
        # the smallest grid of the budget sweep: 24 heads, 8,192 tokens
        _case(name="sweep_8k", H=24, T=8, Hg=32, Wg=32, f8=0.05, f4=0.20),
        # Wan2.1-1.3B-shaped 480p, the ordinary layer call
        _case(name="wan1p3b_480p", H=12, T=21, Hg=30, Wg=52, f8=0.10, f4=0.30),
        # the same with one ranking per head, as the algorithm is printed: rows of unequal length
        _case(name="wan1p3b_480p_head_scope", H=12, T=21, Hg=30, Wg=52, f8=0.10, f4=0.30, head_scope=True),
        # the same on the balanced ragged partition, at a later denoising step whose scales are carried over
        _case(name="wan1p3b_480p_balanced_step", mode="cached", H=12, T=21, Hg=30, Wg=52, f8=0.10, f4=0.30, balanced=True),
        # the same with text tokens in front of the video tokens (they run in bf16, outside the budget)
        _case(name="wan1p3b_480p_prefix", H=12, T=21, Hg=30, Wg=52, f8=0.10, f4=0.30, prefix=226),
        # HunyuanVideo-shaped 720p: the longest sequence, the smallest budget
        _case(name="hunyuan_720p", H=24, T=33, Hg=45, Wg=80, f8=0.05, f4=0.20),
        # Wan2.1-14B-shaped 720p with few-step budgets: the largest ordinary call
        _case(name="wan14b_720p", H=40, T=21, Hg=45, Wg=80, f8=0.20, f4=0.40, k_outliers=True),
        # the same with the bf16 tier as the high one and the 8-bit tier as the low one: the largest call
        _case(name="wan14b_720p_hi", H=40, T=21, Hg=45, Wg=80, f16=0.20, f8=0.40, k_outliers=True),
        # layer inputs and outputs in pinned host memory (a model whose activations are offloaded)
        _case(name="host_480p", mode="host", H=12, T=21, Hg=30, Wg=52, f8=0.10, f4=0.30),
        # the draft map alone: two heads at 480p, for a caller that may not allocate
        _case(name="draft_map", mode="map", H=2, T=21, Hg=30, Wg=52),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_BUDGETS = ((0.0, 0.05, 0.20), (0.0, 0.10, 0.30), (0.0, 0.10, 0.40), (0.0, 0.20, 0.40), (0.0, 0.25, 0.25),
            (0.0, 0.20, 0.60), (0.0, 0.0, 0.40), (0.0, 0.20, 0.0), (0.15, 0.25, 0.30), (0.20, 0.40, 0.0),
            (0.10, 0.0, 0.30))


def _blocks(c):
    """Key blocks of one head."""
    if c["balanced"]:
        return c["T"] * -(-c["Hg"] * c["Wg"] // 64)
    return c["T"] * -(-c["Hg"] // 8) * -(-c["Wg"] // 8)


def _pairs(c):
    """Retained pairs of 64-token blocks over all heads (bf16 pairs, prefix pairs among them, counted twice)."""
    R, rp = _blocks(c), -(-c["prefix"] // 64)
    return c["B"] * c["H"] * (R * R * (2 * c["f16"] + c["f8"] + c["f4"]) + 2 * (2 * R * rp + rp * rp))


_MOST = 40 * 1260 ** 2 * 0.6  # pairs of the largest ordinary call


def draw(rng):
    """One more problem: clip lengths 1 to 33 latent frames, frames 16 x 16 to 45 x 80, 1,000 to 120,000 tokens."""
    mode = rng.choice(("call",) * 6 + ("cached", "reuse", "host", "map"))
    while True:
        tokens = _log_int(rng, 1000, 118800)
        Hg, Wg = rng.randint(16, 45), rng.randint(16, 80)
        T = max(1, round(tokens / (Hg * Wg)))
        if T <= 33 and T * Hg * Wg <= 118800:
            break
    c = _case(mode=mode, H=_log_int(rng, 1, 40), d=rng.choice((128, 128, 128, 64)), T=T, Hg=Hg, Wg=Wg)
    if mode == "map":
        while c["T"] > 1 and _blocks(c) ** 2 > 1 << 20:
            c["T"] -= 1
        c["H"] = max(1, min(c["H"], (1 << 20) // _blocks(c) ** 2))
        return c
    c["B"] = 2 if rng.random() < 0.15 and c["H"] <= 20 else 1
    c["f16"], c["f8"], c["f4"] = rng.choice(_BUDGETS)
    option = rng.choice(("plain", "plain", "balanced", "head_scope", "prefix"))
    if option == "balanced":
        c["balanced"] = True
    elif option == "head_scope":
        c["head_scope"] = True
    elif option == "prefix" and mode != "host":
        c["prefix"] = rng.randint(20, 512)
    c["k_outliers"] = rng.random() < 0.25
    while _pairs(c) > 0.5 * _MOST and c["H"] > 1:
        c["H"] -= 1
    if mode == "host":  # three states of pinned memory at a time
        c["H"] = max(1, min(c["H"], int(12 * 32760 / (c["B"] * c["T"] * Hg * Wg))))
    return c


def _tensor(c, gen, scale_channels=None):
    """bf16 [B, H, prefix + N, d]: per channel a smooth field over the latent grid plus white noise, as the activations of
    a video model are smooth in space and time; text tokens in front are plain normals."""
    dev, BH, d = "cuda", c["B"] * c["H"], c["d"]
    T, Hg, Wg, P = c["T"], c["Hg"], c["Wg"], c["prefix"]
    N = T * Hg * Wg
    out = torch.empty(BH, P + N, d, dtype=torch.bfloat16, device=dev)
    coarse = (max(2, T // 4 + 1), max(2, Hg // 4 + 1), max(2, Wg // 4 + 1))
    step = max(1, int(2 ** 27 // (N * d)))
    for h in range(0, BH, step):
        n = min(step, BH - h)
        z = torch.randn(n, d, *coarse, generator=gen, device=dev)
        z = F.interpolate(z, size=(T, Hg, Wg), mode="trilinear", align_corners=True).reshape(n, d, N)
        z = z / z.std(dim=2, keepdim=True)
        z = z + 0.5 * torch.randn(n, d, N, generator=gen, device=dev)
        if scale_channels is not None:
            z = z * scale_channels.view(1, d, 1)
        out[h:h + n, P:] = z.transpose(1, 2).to(torch.bfloat16)
    if P:
        out[:, :P] = torch.randn(BH, P, d, generator=gen, device=dev).to(torch.bfloat16)
    return out.view(c["B"], c["H"], P + N, d)


def prepare(case, seed):
    c = {**_DEFAULTS, **case}
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    BH, d = c["B"] * c["H"], c["d"]
    if c["mode"] == "map":
        R = _blocks(c)
        desc = [torch.randn(BH, R, d, generator=gen, device="cuda") * s for s in (0.7, 0.7, 0.7, 0.7)]
        desc[1] += 2.0  # maxima over a region lie above its mean
        desc[3] += 2.0
        return {"c": c, "desc": desc, "map": torch.empty(BH, R, R, device="cuda")}
    boost = None
    if c["k_outliers"]:  # a few key channels far larger than the rest
        boost = torch.ones(d, device="cuda")
        boost[3::32] = 20.0
    q, k, v = _tensor(c, gen), _tensor(c, gen, boost), _tensor(c, gen)
    budget = (c["f16"], c["f8"], c["f4"])
    grid = (c["B"], c["H"], c["T"], c["Hg"], c["Wg"], d)
    scope = da2.binding.DA2_RANK_HEAD if c["head_scope"] else da2.binding.DA2_RANK_ROW
    part = da2.binding.DA2_PARTITION_BALANCED if c["balanced"] else da2.binding.DA2_PARTITION_TILES
    if c["mode"] == "host":
        pin = [t.cpu().pin_memory() for t in (q, k, v)]
        out = torch.empty_like(pin[0], pin_memory=True)
        return {"c": c, "in": pin, "out": out,
                "pipe": da2.HostPipeline(*grid, *budget, rank_scope=scope, partition=part)}
    plan = da2.da2_plan(*grid, *budget, rank_scope=scope, n_prefix=c["prefix"], partition=part)
    ws = torch.empty(int(plan.info.workspace_bytes), dtype=torch.uint8, device="cuda")
    s = {"c": c, "plan": plan, "q": q, "k": k, "v": v, "ws": ws, "out": torch.empty_like(q)}
    if c["mode"] in ("cached", "reuse"):  # the step before this one, on slightly different activations
        prev = [(t.float() * 0.98).to(torch.bfloat16) for t in (q, k, v)]
        da2.da2_prepare(plan, *prev, ws)
    return s


def run(state):
    s, mode = state, state["c"]["mode"]
    if mode == "map":
        da2.da2_draft_map_noalloc(*s["desc"], 0.2, 1.0 / math.sqrt(s["c"]["d"]), s["map"])
        return s["map"]
    if mode == "host":
        s["pipe"].run(*s["in"], s["out"])
        return s["out"]
    plan, q, k, v, ws, out = s["plan"], s["q"], s["k"], s["v"], s["ws"], s["out"]
    if mode == "call":
        da2.attention(plan, q, k, v, workspace=ws, out=out)
        return out
    if mode == "cached":
        da2.da2_prepare_cached_scales(plan, q, k, v, ws, reselect=True)
    else:
        da2.da2_refresh_operands(plan, q, k, v, ws)
    da2.da2_attention_fwd(plan, q, k, v, ws, out)
    return out


def work(case):
    """Q, K, V read and the output written once; two products for each retained pair of valid tokens, and the draft map's
    two contractions."""
    c = {**_DEFAULTS, **case}
    BH, d, R, P = c["B"] * c["H"], c["d"], _blocks(c), c["prefix"]
    N = c["T"] * c["Hg"] * c["Wg"]
    if c["mode"] == "map":
        return {"bytes": BH * (4 * R * d + R * R) * 4, "flops": 4 * BH * R * R * d}
    kept = c["f16"] + c["f8"] + c["f4"]
    flops = 4 * BH * d * (N * (N * kept + P) + P * (N + P))
    if c["mode"] != "reuse":
        flops += 4 * BH * R * R * d
    return {"bytes": 4 * BH * (P + N) * d * 2, "flops": flops}


def tolerance(case):
    # the map is a softmax of fp32 descriptors; the outputs are bf16, of products in bf16, 8-bit and 4-bit formats
    return {"rel": 1e-5} if case.get("mode") == "map" else {"rel": 1e-2}
