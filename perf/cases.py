"""The work a user of this framework has it do, as measurable cases: rounds of draft-and-verify over the
grids, vocabularies and sampling rules of the repository's own workloads and tests, the four stages called
one by one, the drafter's draw, the islands of the redraw, and a whole speculative round with its redraw.

Every case is a dict of plain values.  ``prepare`` makes the logits (the repository's synthetic recipe), the
draft tokens and the buffers a serving program keeps; ``run`` makes the calls such a program makes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_05149_b200 import binding, synth

_CFG = ("B", "H", "W", "V", "r", "dtype", "sigma", "cfg_scale", "temperature", "top_k", "pool_k", "pool_delta",
        "radius", "clip_before_first", "accept_mode", "tau", "resample_mode")


def _case(name, path, cfg=None, **over):
    base = cfg if cfg is not None else synth.RoundConfig(name, B=1, H=16, W=16, V=4096)
    c = {k: over.get(k, getattr(base, k)) for k in _CFG}
    c.update({k: v for k, v in over.items() if k not in c})
    return dict(name=name, path=path, **c)


def listed():
    C = synth.CONFIGS
    return [
        # the smallest call: one 256-token image, fp32 logits, no top-k cut -- launches and latency
        _case("round_16x16_f32", "round", C["C1"]),
        # one 512-pixel image with the paper's probability pooling and a top-k cut, batch 1 (interactive use)
        _case("round_32x32_pooled", "round", C["C2"]),
        # a small serving batch of 1024-pixel images: CFG and top-k, narrow window
        _case("round_64x64_b8", "round", C["C3"]),
        # the headline workload: batch 32, CFG, top-k, three expansion rounds
        _case("round_64x64_b32", "round", C["C4"]),
        # the paper's default sampling (no cut, CFG 4, pooling, the relaxed rule of Eq. 5, target redraws)
        _case("default_64x64_b16", "round", C["P4"], B=16),
        # the same sampling under Eq. 1: residual redraws over the whole vocabulary
        _case("default_eq1_64x64_b4", "round", C["P4"], B=4, accept_mode=0, resample_mode=0),
        # a larger grid with the smaller codebook, target close to the draft (the sweep's 96 x 96 points)
        _case("round_96x96_v8192", "round", C["C4"], B=4, H=96, W=96, V=8192, sigma=0.1, radius=1),
        # a non-square grid, ratio 3, a vocabulary that splits evenly over nothing, fp32, no guidance, T != 1
        _case("round_ragged_f32", "round", B=3, H=36, W=51, V=12296, r=3, dtype="f32", top_k=1000, sigma=1.0,
              temperature=0.9, radius=2, resample_mode=3),
        # a host that runs the four stages itself (it looks at the masks in between)
        _case("stages_64x64_b2", "stages", C["C4"], B=2),
        # step 1 of a round: the drafter's draw for a batch of 32
        _case("draft_32x32_b32", "draft", C["C4"]),
        # a whole speculative round: draft draw, round, islands, schedule, step-by-step redraw, prefix
        _case("loop_64x64_b4", "loop", C["C4"], B=4, window=16),
        # scheduling alone: islands and steps of a batch of sparse rejection masks
        _case("islands_64x64_b32", "islands", C["C4"], density=0.02, window=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["round"] * 6 + ["default"] * 4 + ["stages"] * 2 + ["draft"] * 3 + ["loop"] * 2 + ["islands"] * 2)
    r = rng.choice([2, 2, 2, 2, 1, 3, 4])
    h, w = _log_int(rng, 16, 96) // r, _log_int(rng, 16, 96) // r
    # codebooks are powers of two or multiples of 1024 in earnest; sizes in between are allowed
    V = rng.choice([4096, 8192, 16384, 16384, 8 * _log_int(rng, 256, 4096), 1024 * rng.randint(2, 20)])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    cfg_scale = rng.choice([0.0, 1.5, 3.0, 3.0, 4.0, 7.5])
    top_k = 0 if path == "default" else max(16, int(V * rng.choice([1 / 16, 1 / 8, 1 / 8, 1 / 5])))
    if path == "draft" and rng.random() < 0.3:
        top_k = 0
    pool = path == "default" and rng.random() < 0.6 or path == "round" and rng.random() < 0.2
    eq5 = path == "default" and rng.random() < 0.5
    row = V * (2 if dtype == "bf16" else 4) * (1 if path == "draft" or not cfg_scale else 2)
    limit = 2.0e9 if path in ("round", "default", "draft") else 0.5e9   # bytes of logits
    n = h * w * (1 if path == "draft" else r * r)
    most = 64 if path == "islands" else max(1, min(64, int(limit / (row * n))))
    c = _case("drawn", "round" if path == "default" else path, B=_log_int(rng, 1, most), H=h * r, W=w * r, V=V, r=r, dtype=dtype,
              sigma=rng.choice([0.1, 0.5, 1.0, 2.0]), cfg_scale=cfg_scale,
              temperature=rng.choice([1.0, 1.0, 1.0, round(rng.uniform(0.7, 1.3), 2)]), top_k=top_k,
              pool_k=min(rng.choice([100, 500, 1000]), V // 4) if pool else 1, pool_delta=rng.choice([0.05, 0.1, 0.3]),
              radius=rng.randint(1, 3), accept_mode=1 if eq5 else 0, tau=1e-4,
              resample_mode=2 if eq5 else rng.choice([0, 0, 3, 1]))
    if path == "islands":
        c["density"] = rng.choice([0.002, 0.01, 0.05])
    if path in ("islands", "loop"):
        c["window"] = rng.choice([8, 16])
    del c["name"]
    return c


def _config(case, seed):
    return synth.RoundConfig("case", seed=seed, **{k: case[k] for k in _CFG})


def _draft_tokens(cfg, draft, gen):
    """One draw per low-res cell from the draft distribution (temperature, top-k), by the Gumbel rule."""
    tok = torch.empty((cfg.B, cfg.h, cfg.w), dtype=torch.int32, device=draft.device)
    inv_t = float(np.float32(1.0) / np.float32(cfg.temperature))
    for b in range(cfg.B):
        z = draft[b].float() * inv_t
        g = torch.rand(z.shape, generator=gen, device=z.device).clamp_min_(1e-12).log_().neg_().log_().neg_()
        if 0 < cfg.top_k < cfg.V:
            theta = torch.topk(z, cfg.top_k, dim=-1, sorted=False).values.amin(-1, keepdim=True)
            z.masked_fill_(z < theta, -math.inf)
        tok[b] = g.add_(z).argmax(-1).to(torch.int32)
    return tok


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    cfg = _config(case, seed)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 2_000_003 + 17)
    p = binding.params_from_config(cfg)
    ctx = binding.Context(dev.index)
    ctx.ensure_workspace(p)
    B, H, W, h, w = cfg.B, cfg.H, cfg.W, cfg.h, cfg.w
    i32 = dict(dtype=torch.int32, device=dev)
    f32 = dict(dtype=torch.float32, device=dev)
    s = dict(path=case["path"], p=p, ctx=ctx, window=case.get("window", 16), max_step=H * W)
    path = case["path"]

    if path == "islands":     # R_X of sparse random rejections
        hits = torch.rand((B, H, (W + 31) // 32, 32), generator=gen, device=dev) < case["density"]
        hits = hits & (torch.arange(hits.shape[2] * 32, device=dev).view(1, 1, -1, 32) < W)
        words = (hits.to(torch.int64) << torch.arange(32, device=dev)).sum(-1)
        reject = torch.where(words >= 2 ** 31, words - 2 ** 32, words).to(torch.int32).contiguous()
        s["expand"] = torch.empty_like(reject)
        ctx.mulo_local_reject_expand(p, reject, torch.zeros((B,), **i32), s["expand"], torch.empty((B,), **i32))
        s["tokens"] = torch.randint(0, cfg.V, (B, h, w), generator=gen, **i32).repeat_interleave(cfg.r, 1) \
            .repeat_interleave(cfg.r, 2).contiguous()
    elif path == "draft":
        s["draft_lo"] = torch.empty((B, h, w, cfg.V), dtype=cfg.torch_dtype, device=dev)
        for b in range(B):
            s["draft_lo"][b] = 2.0 * torch.randn((h, w, cfg.V), generator=gen, **f32)
    else:
        s.update(synth.build_batch(cfg, dev))
        s["tok_lo"] = torch.empty((B, h, w), **i32) if path == "loop" else _draft_tokens(cfg, s["draft_lo"], gen)
    if path in ("round", "stages", "loop"):
        s["out"] = binding.alloc_round_outputs(p, dev, probs=path != "loop")
    if path == "stages":
        s.update(tok_hi=torch.empty((B, H, W), **i32), stats=torch.empty((B, h, w, 4), **f32),
                 q_hi=torch.empty((B, H, W), **f32))
    if path in ("loop", "draft", "islands"):
        s.setdefault("tok_lo", torch.empty((B, h, w), **i32))
    if path in ("loop", "islands"):
        s.update(labels=torch.empty((B, H, W), **i32), n_islands=torch.empty((B,), **i32),
                 step=torch.empty((B, H, W), **i32), n_steps=torch.empty((B,), **i32),
                 prefix=torch.empty((B, h, w), **i32), rows=torch.empty((B, 256, 2), **i32),
                 size=torch.empty((B, 256), **i32))
    if path == "loop":
        s.update(pos_list=torch.empty((B * H * W,), **i32), offsets=torch.empty((2 * (H * W + 2),), **i32))
    return s


def run(s):
    ctx, p, path = s["ctx"], s["p"], s["path"]
    if path == "round":
        o = s["out"]
        ctx.mulo_round(p, s["cond"], s["uncond"], s["draft_lo"], s["tok_lo"], s["nn"], o["out_tok"],
                       o["reject_bits"], o["expand_bits"], o["p_tok"], o["q_tok"], o["accept_prob"],
                       o["n_reject"], o["n_expand"], o["first_reject"])
        return o
    if path == "stages":
        o = s["out"]
        ctx.mulo_upsample_pool(p, s["draft_lo"], s["tok_lo"], s["nn"], s["tok_hi"], s["stats"], s["q_hi"])
        ctx.mulo_verify(p, s["cond"], s["uncond"], s["draft_lo"], s["stats"], s["tok_hi"], s["nn"], o["p_tok"],
                        o["q_tok"], o["accept_prob"], o["reject_bits"], o["n_reject"], o["first_reject"])
        ctx.mulo_local_reject_expand(p, o["reject_bits"], o["first_reject"], o["expand_bits"], o["n_expand"])
        ctx.mulo_resample(p, s["cond"], s["uncond"], s["draft_lo"], s["stats"], s["tok_hi"], s["nn"],
                          o["reject_bits"], o["expand_bits"], o["out_tok"])
        return dict(o, tok_hi=s["tok_hi"], stats=s["stats"], q_hi=s["q_hi"])
    if path == "draft":
        ctx.mulo_sample_draft(p, s["draft_lo"], s["tok_lo"])
        return s["tok_lo"]
    if path == "islands":
        ctx.mulo_islands(p, s["expand"], s["labels"], s["n_islands"], s["rows"], s["size"])
        ctx.mulo_island_schedule(p, s["labels"], s["window"], s["step"], s["n_steps"])
        ctx.mulo_downsample(p, s["tokens"], s["prefix"])
        return {k: s[k] for k in ("labels", "n_islands", "rows", "size", "step", "n_steps", "prefix")}
    # a whole speculative round; the redraw's length is the one thing the host reads
    o = s["out"]
    ctx.mulo_sample_draft(p, s["draft_lo"], s["tok_lo"])
    ctx.mulo_round(p, s["cond"], s["uncond"], s["draft_lo"], s["tok_lo"], s["nn"], o["out_tok"], o["reject_bits"],
                   o["expand_bits"], None, None, None, o["n_reject"], o["n_expand"], o["first_reject"])
    ctx.mulo_islands(p, o["expand_bits"], s["labels"], s["n_islands"])
    ctx.mulo_island_schedule(p, s["labels"], s["window"], s["step"], s["n_steps"])
    nfe = int(s["n_steps"].max().item())
    ctx.mulo_redraw_plan(p, s["step"], s["max_step"], s["pos_list"], s["offsets"])
    for k in range(1, nfe + 1):
        ctx.mulo_redraw_step(p, k, s["max_step"], s["pos_list"], s["offsets"], s["cond"], s["uncond"], o["out_tok"])
    ctx.mulo_downsample(p, o["out_tok"], s["prefix"])
    return dict(tok_lo=s["tok_lo"], out_tok=o["out_tok"], reject_bits=o["reject_bits"], expand_bits=o["expand_bits"],
                labels=s["labels"], step=s["step"], prefix=s["prefix"])


def work(case):
    cfg = _config(case, 0)
    n, cells, esz = cfg.B * cfg.H * cfg.W, cfg.B * cfg.h * cfg.w, cfg.elem_size
    rows = (2 if cfg.has_uncond else 1) * n          # target logit rows
    mix = (3 if cfg.has_uncond else 0) + 2           # guidance mix, exponent and sum per vocabulary entry
    masks = 2 * cfg.B * cfg.H * ((cfg.W + 31) // 32) * 4
    path = case["path"]
    if path == "islands":
        return {"bytes": masks // 2 + n * 4 * 3 + cells * 4 + cfg.B * 256 * 12, "flops": 0}
    if path == "draft":
        return {"bytes": cells * (cfg.V * esz + 4), "flops": cells * cfg.V * 2}
    round_bytes = cfg.algorithmic_bytes_per_position() * n + cells * 4 + masks
    flops = n * cfg.V * mix + cells * cfg.V * 2
    if path == "round":
        return {"bytes": round_bytes, "flops": flops}
    if path == "stages":       # the masks are the host's to look at, so the target rows are read by two calls
        return {"bytes": round_bytes + rows * cfg.V * esz + cells * cfg.V * esz * 2 + cells * 16 + n * 12,
                "flops": 2 * flops + cells * cfg.V * 2}
    # the whole round: the draft logits once more for the draft's draw, every redrawn row once more
    return {"bytes": round_bytes + cells * cfg.V * esz + rows * cfg.V * esz + n * 4 * 6,
            "flops": 2 * flops}


def tolerance(case):
    if case["path"] == "islands":
        return "exact"
    # Tokens: an inverse-CDF draw comes out differently only where its uniform falls between two correct
    # implementations' CDF edges (a few 1e-8 of mass per edge, one edge per active token): 6e-5 of the draws
    # at top-k 2000 between two of the kernels, 2.4e-4 over 16384 tokens against the fp64 oracle; small grids
    # may see one or two.  Probabilities: sums of up to V fp32 exponentials in another order, 3e-7 (largest
    # 8e-7) between two of the kernels.
    n = case["B"] * case["H"] * case["W"]
    draws = n // (case["r"] ** 2) if case["path"] in ("draft", "loop") else n
    differ = min(0.01, max(2.5e-4 if case["top_k"] else 1e-3, 2.5 / draws))
    return {"rel": 2e-6, "max": 1e-5, "differ": differ}
