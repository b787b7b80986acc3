"""Performance cases of the cached DiT denoising step, through the package's public entry points.

Each case is one thing a user of the library has it do, at one size.  Three kinds:

  step      `Hero.hero_step` (or `hero_step_host` on pinned host buffers) of a whole model.  `mode` says which
            part of the denoising schedule one pass is: "cached" (one step between two full ones: select and
            refresh in the shallow blocks, extrapolation in the deep ones), "full" (every row of every block,
            what fills the caches) or "interval" (one full step and the cached steps up to the next).
  block     one block of the model: `hero_select_tokens` + `hero_refresh_block` on the drawn rows (mode
            "cached") or `hero_refresh_block` on all rows (mode "full").
  features  the stateless kernels on one layer's feature cache: gather of the selected rows, LayerNorm with
            modulation of the gathered rows, scatter back, linear extrapolation and its error measure.

Inputs follow the synthetic recipe of the repository's workloads: weights and biases N(0, 0.02^2), tokens and
timestep embeddings N(0, 1), feature histories A and A + 0.1 B; everything is made on the device from the seed.
"""
import math

import torch

import paper_2508_17588_b200 as H

# What a case does not name.  The base block: head dimension 64, four modulation vectors, 2x2 patches, a quarter
# of the tokens refreshed, two warm-up full steps.
_BASE = dict(kind="step", mode="cached", host=0, dtype="bf16", head_dim=64, batch=2, n_text=226, patch_h=2, patch_w=2,
             ratio_num=1, ratio_den=4, quota_mode=0, full_interval=5, has_gate=0, deep_collapse=0,
             track_mode=0, share_selection=0, attend_mode=0, qk_norm=0, rope=0)
# The 5-billion-parameter video DiT block of the repository's workloads: 48 heads, 13 latent frames of 30 x 45 tokens.
_VIDEO = dict(_BASE, hidden=3072, ffn_dim=12288, temb_dim=512, frames=13, grid_h=30, grid_w=45)


def listed():
    return [
        # The smallest model, in fp32: what somebody checks an integration with.  About 25 launches of a few
        # microseconds each; latency is all there is.
        dict(_BASE, name="tiny_fp32", dtype="fp32", n_blocks=4, n_shallow=2, hidden=128, ffn_dim=512, temb_dim=128,
             batch=1, frames=2, grid_h=8, grid_w=8, n_text=16, full_interval=0),
        # A whole fp32 model of moderate width: numerics runs, where bf16 rounding would hide what is looked for.
        dict(_BASE, name="width512_fp32", dtype="fp32", n_blocks=6, n_shallow=2, hidden=512, ffn_dim=2048, temb_dim=256,
             frames=3, grid_h=18, grid_w=23, n_text=77),
        # The 42-block schedule in miniature (307 rows, odd grid), one full step and four cached ones: the smallest
        # bf16 model, launch after launch.
        dict(_BASE, name="mini42_interval", mode="interval", n_blocks=42, n_shallow=14, hidden=256, ffn_dim=768,
             temb_dim=64, frames=3, grid_h=9, grid_w=11, n_text=10),
        # A small image-sized model (one frame, a single sequence, gates, rotary embedding, one list for all blocks),
        # cached step: a few hundred refreshed rows per block.
        dict(_BASE, name="width768_cached", n_blocks=12, n_shallow=4, hidden=768, ffn_dim=3072, temb_dim=256, batch=1,
             frames=1, grid_h=33, grid_w=45, n_text=77, has_gate=1, rope=1, share_selection=1),
        # A medium video model with the guidance pair, cached step.
        dict(_BASE, name="width1024_cached", n_blocks=24, n_shallow=8, hidden=1024, ffn_dim=4096, temb_dim=256,
             frames=5, grid_h=18, grid_w=31, n_text=120),
        # The same size class with every row computed (and a width that is no power of two): the full step of a
        # collapsed deep stack.
        dict(_BASE, name="width1152_full", mode="full", n_blocks=16, n_shallow=6, hidden=1152, ffn_dim=4608, temb_dim=384,
             frames=5, grid_h=17, grid_w=30, n_text=77, deep_collapse=1, ratio_num=1, ratio_den=5),
        # One block of the 5B model at a refresh ratio of 10 %: the low end of the refresh sweep.
        dict(_VIDEO, name="block_refresh10", kind="block", n_blocks=1, n_shallow=1, full_interval=0, ratio_num=1,
             ratio_den=10),
        # The same block with all 17776 rows: one forty-second of a full step.
        dict(_VIDEO, name="block_full", kind="block", mode="full", n_blocks=1, n_shallow=1, full_interval=0),
        # The headline: cached step of the 42-block model, 14 blocks refreshed at 25 %, 28 extrapolated.
        dict(_VIDEO, name="dit42_cached", n_blocks=42, n_shallow=14),
        # Reconstruction setting of the method (one sequence, 2x3 patches, one token of each, 20 blocks refreshed, full
        # step every second one), from pinned host buffers to pinned host buffers.
        dict(_VIDEO, name="recon_host", host=1, n_blocks=42, n_shallow=20, batch=1, frames=11, patch_w=3, ratio_num=1,
             ratio_den=5, quota_mode=1, full_interval=2),
        # The base model's own block (per-head q/k norm, rotary embedding, gates) under the literal reading of the
        # refresh: queries see the refreshed rows and the text only, strict oldest-first tracking.
        dict(_VIDEO, name="base_block_literal", n_blocks=12, n_shallow=6, frames=9, grid_w=44, qk_norm=1, rope=1,
             has_gate=1, attend_mode=1, track_mode=1),
        # One layer's feature cache at full size, 10 % of the rows: the memory-bound kernels and the layer analysis.
        dict(_VIDEO, name="features_10", kind="features", ratio_num=1, ratio_den=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _tokens(rng, lo, hi):
    """frames, grid_h, grid_w with about `lo`..`hi` tokens in all, uneven sides included."""
    n = _log(rng, lo, hi)
    frames = rng.choice([1, 2, 3, 5, 7, 9, 11, 13])
    while frames > 1 and n / frames < 20:
        frames -= 1
    side = math.sqrt(n / frames)
    grid_h = max(3, int(side * rng.uniform(0.65, 0.95)))
    return dict(frames=frames, grid_h=grid_h, grid_w=max(4, int(n / frames / grid_h)))


def _selection(rng):
    num, den = rng.choice([(1, 10), (1, 5), (1, 4), (1, 4), (1, 3), (1, 2)])
    ph, pw = rng.choice([(2, 2), (2, 2), (2, 3)])
    return dict(patch_h=ph, patch_w=pw, ratio_num=num, ratio_den=den, quota_mode=rng.choice([0, 0, 1]) if den <= 5 else 0,
                track_mode=rng.choice([0, 0, 1]), full_interval=rng.choice([2, 3, 5]))


def draw(rng):
    while True:                                      # at most the work of the largest listed case
        case = _draw(rng)
        if work(case)["flops"] <= 5e13:
            return case


def _draw(rng):
    family = rng.choice(["fp32", "small", "small", "medium", "medium", "large", "block", "features"])
    case = dict(_BASE, **_selection(rng))
    case.update(batch=rng.choice([1, 2, 2]), n_text=rng.choice([0, 7, 16, 77, 120, 226]))
    if family == "features":
        case.update(kind="features", hidden=64 * int(_log(rng, 4, 48)), dtype=rng.choice(["bf16", "bf16", "fp32"]))
        case.update(_tokens(rng, 500, 17550 if case["dtype"] == "bf16" else 8000), temb_dim=64, n_text=226)
        return case
    if family == "fp32":
        case.update(dtype="fp32", hidden=64 * int(_log(rng, 1, 9)), temb_dim=rng.choice([64, 128, 256]),
                    n_blocks=rng.randint(2, 6), mode=rng.choice(["cached", "cached", "full"]), **_tokens(rng, 100, 1300))
        case["ffn_dim"] = 4 * case["hidden"]
    elif family == "block":
        case.update(kind="block", hidden=64 * int(_log(rng, 16, 49)), temb_dim=512, n_blocks=1, n_shallow=1,
                    mode=rng.choice(["cached", "cached", "full"]), n_text=226, **_tokens(rng, 2000, 17550))
        case["ffn_dim"] = 4 * case["hidden"]
        return case
    else:
        width, rows, blocks = {"small": ((2, 12), (100, 2000), (4, 42)), "medium": ((10, 26), (800, 6000), (4, 24)),
                               "large": ((32, 49), (4000, 17550), (2, 8))}[family]
        case.update(hidden=64 * int(_log(rng, *width)), temb_dim=rng.choice([64, 256, 512]),
                    n_blocks=int(_log(rng, *blocks)), mode=rng.choice(["cached", "cached", "cached", "full", "interval"]),
                    host=rng.choice([0, 0, 0, 1]), **_tokens(rng, *rows))
        case["ffn_dim"] = case["hidden"] * rng.choice([3, 4, 4])
        case.update(has_gate=rng.choice([0, 1]), rope=rng.choice([0, 0, 1]), qk_norm=rng.choice([0, 0, 1]),
                    deep_collapse=rng.choice([0, 0, 0, 1]), share_selection=rng.choice([0, 0, 0, 1]),
                    attend_mode=rng.choice([0, 0, 0, 1]))
    case["n_shallow"] = max(1, int(case["n_blocks"] * rng.choice([0.33, 0.33, 0.5])))
    return case


# ---------------------------------------------------------------------------------------------------------------
def _rows(case):
    """Video tokens and sequence length."""
    v = case["frames"] * case["grid_h"] * case["grid_w"]
    return v, v + case["n_text"]


def _n_sel(case):
    """Rows a cached step refreshes, up to the rounding of one call."""
    v, _ = _rows(case)
    if case["quota_mode"] == 0:
        return v * case["ratio_num"] // case["ratio_den"]
    total = 0
    for y in range(0, case["grid_h"], case["patch_h"]):
        for x in range(0, case["grid_w"], case["patch_w"]):
            n = min(case["patch_h"], case["grid_h"] - y) * min(case["patch_w"], case["grid_w"] - x)
            total += min(n, (2 * n * case["ratio_num"] + case["ratio_den"]) // (2 * case["ratio_den"]))
    return total * case["frames"]


class _Maker:
    """Normal tensors from one seed, in the order they are asked for."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.dtype = torch.bfloat16 if dtype == "bf16" else torch.float32

    def __call__(self, *shape, std=1.0, mean=0.0, dtype=None):
        return torch.empty(shape, dtype=dtype or self.dtype, device="cuda").normal_(mean, std, generator=self.g)


def _weights(case, make):
    D, F, E = case["hidden"], case["ffn_dim"], case["temb_dim"]
    n_mod = 6 if case["has_gate"] else 4
    shapes = dict(w_mod=(n_mod * D, E), b_mod=(n_mod * D,), w_qkv=(3 * D, D), b_qkv=(3 * D,), w_o=(D, D), b_o=(D,),
                  w_1=(F, D), b_1=(F,), w_2=(D, F), b_2=(D,))
    w = {name: make(*shape, std=0.02) for name, shape in shapes.items()}
    if case["qk_norm"]:
        w.update(qn_w=make(64, std=0.1, mean=1.0), qn_b=make(64, std=0.1), kn_w=make(64, std=0.1, mean=1.0),
                 kn_b=make(64, std=0.1))
    return w


def _config(case, seed):
    cfg = {k: v for k, v in case.items() if k not in ("name", "kind", "mode", "host")}
    cfg.update(n_heads=case["hidden"] // case["head_dim"], warmup_full_steps=2, seed=seed)
    return cfg


def prepare(case, seed):
    """Weights, context with its caches filled by the warm-up full steps, the step's tokens and embeddings."""
    make = _Maker(seed, case["dtype"])
    B, D, E = case["batch"], case["hidden"], case["temb_dim"]
    video, N = _rows(case)
    s = dict(case=case)
    if case["kind"] == "features":
        # The list comes from the library's own sampler on the same token grid (a one-head model carries it).
        c = dict(case, n_blocks=1, n_shallow=1, hidden=64, ffn_dim=64)
        hero = H.Hero(_config(c, seed), [_weights(c, make)])
        idx = torch.empty(video, dtype=torch.int32, device="cuda")
        s["idx"] = idx[:hero.hero_select_tokens(0, idx)].clone()
        hero.close()
        n = s["idx"].numel()
        s["x"], s["cache"] = make(B, N, D), make(B, N, D)
        s["g_prev"] = make(B, N, D)
        s["g_last"] = s["g_prev"] + 0.1 * make(B, N, D)
        s["g_true"] = s["g_last"] + 0.1 * make(B, N, D)
        s["shift"], s["scale"] = make(B, D, std=0.3, dtype=torch.float32), make(B, D, std=0.3, dtype=torch.float32)
        s["rows"], s["normed"] = make(B, n, D), make(B, n, D)
        s["predicted"] = torch.empty_like(s["g_last"])
        s["err"] = torch.zeros(2, dtype=torch.float64, device="cuda")
        return s
    hero = s["hero"] = H.Hero(_config(case, seed), [_weights(case, make) for _ in range(case["n_blocks"])])
    s["x0"] = make(B, N, D)
    s["x"] = s["x0"].clone()
    s["temb"] = [make(B, E) for _ in range(8)]
    if case["kind"] == "block":
        s["idx"] = torch.empty(video, dtype=torch.int32, device="cuda")
        s["call"] = 0
        hero.hero_refresh_block(0, s["x"], s["temb"][0])
        return s
    for step in range(2):
        s["x"].copy_(s["x0"])
        hero.hero_step(step, s["x"], s["temb"][step])
    s["step"] = 2
    if case["host"]:
        s["h_x"] = s["x0"].cpu().pin_memory()
        s["h_temb"] = [t.cpu().pin_memory() for t in s["temb"]]
    return s


def _one_step(s, step):
    """One denoising step: this step's tokens into x, then the model, in place."""
    if s["case"]["host"]:
        # The host buffer carries the sequence on from step to step, as a sampler's does.
        s["hero"].hero_step_host(step, s["h_x"], s["h_temb"][step % 8])
        return s["h_x"]
    s["x"].copy_(s["x0"])
    s["hero"].hero_step(step, s["x"], s["temb"][step % 8])
    return s["x"]


def run(s):
    case = s["case"]
    if case["kind"] == "features":
        H.hero_gather_rows(s["cache"], s["idx"], s["rows"])
        H.hero_gather_ln_modulate(s["x"], s["cache"], s["idx"], s["shift"], s["scale"], s["normed"])
        H.hero_scatter_rows(s["normed"], s["idx"], s["x"])
        H.hero_extrapolate(s["g_prev"], s["g_last"], s["predicted"], 3, 5)
        s["err"].zero_()
        H.hero_extrapolation_error(s["g_prev"], s["g_last"], s["g_true"], 3, 5, s["err"])
        return {"rows": s["rows"], "normed": s["normed"], "x": s["x"], "predicted": s["predicted"], "err": s["err"]}
    hero = s["hero"]
    if case["kind"] == "block":
        s["x"].copy_(s["x0"])
        s["call"] += 1
        temb = s["temb"][s["call"] % 8]
        if case["mode"] == "full":
            hero.hero_refresh_block(0, s["x"], temb)
            return {"x": s["x"]}
        n = hero.hero_select_tokens(0, s["idx"])
        hero.hero_refresh_block(0, s["x"], temb, s["idx"], n)
        return {"x": s["x"], "idx": s["idx"][:n]}
    every = case["full_interval"] or 9
    if case["mode"] == "cached":                     # round and round the steps between two full ones
        out = _one_step(s, s["step"])
        s["step"] = s["step"] + 1 if s["step"] < every else 2
        return {"x": out}
    first = s["step"] + (1 - s["step"]) % every      # the next full step
    last = first if case["mode"] == "full" else first + every - 1
    for step in range(first, last + 1):
        out = _one_step(s, step)
    s["step"] = last + 1
    return {"x": out}


# ---------------------------------------------------------------------------------------------------------------
def work(case):
    e = 2 if case["dtype"] == "bf16" else 4
    B, D = case["batch"], case["hidden"]
    _, N = _rows(case)
    n = _n_sel(case)
    x, sel = B * N * D, B * n * D
    if case["kind"] == "features":
        # rows out of the cache and into the compact copy; rows of x and the cache in, normalised rows out;
        # those into x again; two histories in, prediction out; three tensors into two sums
        return {"bytes": e * (2 * sel + 3 * sel + 2 * sel + 3 * x + 3 * x) + 4 * 4 * n, "flops": 0}
    F, E = case["ffn_dim"], case["temb_dim"]
    L, K = case["n_blocks"], case["n_shallow"]
    n_mod = 6 if case["has_gate"] else 4
    w = 4 * D * D + 2 * D * F + n_mod * D * E + (5 + n_mod) * D + F

    def block(rows, keys):
        return 2 * B * rows * (4 * D * D + 2 * D * F) + 4 * B * rows * keys * D

    keys = case["n_text"] + n if case["attend_mode"] else N
    # Cached step.  Weights of the shallow blocks; K and V of the keys that were not just computed, the branch caches
    # of the other rows; what is refreshed, written; the deep histories; x in and out once.
    refresh = w + 2 * B * (keys - n) * D + 2 * (x - sel) + 4 * sel
    deep = L - K
    histories = 2 * x * 4 / e * bool(deep) if case["deep_collapse"] else 4 * x * deep
    cached = dict(bytes=e * (K * refresh + histories + 2 * x), flops=K * block(n, keys))
    # Full step.  All weights; K, V and both branches of the shallow blocks, the branches (or their sum) of the deep
    # ones written; x in and out once.
    kept = x * 4 / e * bool(deep) if case["deep_collapse"] else 2 * x * deep
    full = dict(bytes=e * (L * w + 4 * x * K + kept + 2 * x), flops=L * block(N, N))
    if case["mode"] == "interval":
        c = case["full_interval"] - 1
        return {k: full[k] + c * cached[k] for k in full}
    return full if case["mode"] == "full" else cached


def tolerance(case):
    """About four times the distance of a pass from the same steps in float64 (caches filled on both sides by their
    own full steps).  fp32: 1.4e-6 (largest element 9e-6 of the rms) at width 512, six blocks.  bf16: 4.5e-3 at 12
    blocks, 7.9e-3 at 8 blocks of width 3072, 9.8e-3 (largest element 0.057) at 42: the residual stream is rounded
    once per block, so the distance goes with the root of the depth.  Feature kernels: one rounding each, of which
    another order of the fp32 sums flips few (2e-5)."""
    if case["kind"] == "features":
        return {"rel": 1e-4, "max": 1e-2} if case["dtype"] == "bf16" else {"rel": 1e-6, "max": 1e-5}
    if case["dtype"] == "fp32":
        return {"rel": 6e-6, "max": 4e-5}
    return {"rel": min(2e-2, 7.5e-3 * math.sqrt(case["n_blocks"])), "max": 0.25}
