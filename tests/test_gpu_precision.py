"""How far probabilities are from 64 bits, against the oracle's doubles: what the fp32 weights and their sums cost beyond the
rounding of the outputs themselves."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2601_05149_b200 import binding, synth

import parity_util as pu

pytestmark = pytest.mark.gpu

BASE = synth.RoundConfig("precision", B=1, H=32, W=32, V=12296, dtype="bf16", sigma=1.0, cfg_scale=3.0, seed=901)


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    binding.lib()
    c = binding.Context(0)
    yield c
    c.close()


def relative(got, want):
    sel = want > 1e-30
    return np.abs(got[sel].astype(np.float64) - want[sel]) / want[sel]


@pytest.mark.parametrize("over", [
    dict(), dict(pool_k=50), dict(top_k=1537), dict(V=16384, top_k=2048, pool_k=50), dict(V=16384, top_k=2048),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "plain")
def test_token_probabilities(ctx, over):
    """Rounding p and q to fp32 makes a mean relative error of 0.36 * 2^-24; the weights' own (2^-22 each, averaged out in the
    sums) and that of their exponents' constant (1.3e-8 times the distance from the maximum at which the mass lies) may come to as
    much again."""
    cfg = dataclasses.replace(BASE, **over)
    batch = pu.build_batch(cfg)
    g = pu.gpu_round(ctx, cfg, batch)
    o = pu.oracle_images(cfg, batch, [0])[0]
    for k in ("p_tok", "q_tok"):
        e = relative(g[k][0], o[k])
        assert e.mean() < 2 * 0.36 * 2.0 ** -24, f"{k}: mean {e.mean():.2e}, largest {e.max():.2e}"


@pytest.mark.parametrize("V,top_k", [(264, 0), (264, 33), (1032, 0), (16384, 2048)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_draft_sums(ctx, dtype, V, top_k):
    """Z_q as mulo_upsample_pool hands it on (an fp32 pair, so that the pair's rounding does not count): fp32 weights of one unit
    in the last place, added in double.  A quarter of one such unit is what is left on average even of 264 weights, of which
    a few hold most of the mass."""
    cfg = dataclasses.replace(BASE, V=V, top_k=top_k, dtype=dtype, temperature=0.8, cfg_scale=0.0)
    batch = pu.build_batch(cfg)
    stats = pu.gpu_stages(ctx, cfg, batch)["stats"][0].astype(np.float64)
    want = orc.upsample_pool_image(pu.orc_params(cfg, 0), synth.to_numpy_logits(batch["draft_lo"][0]),
                                   batch["tok_lo"][0].cpu().numpy())["stats"]
    e = relative(stats[..., 2] + stats[..., 3], want[..., 2])
    assert e.mean() < 2.0 ** -26, f"mean {e.mean():.2e}, largest {e.max():.2e}"


@pytest.mark.parametrize("V,top_k,dtype", [(4096, 512, "f32"), (8192, 2600, "f32"), (16384, 2000, "f32")])
def test_redraws_near_the_draft(ctx, V, top_k, dtype):
    """A target within 0.003 of its draft: the residual is a difference of nearly equal probabilities and has 0.1 % of their mass, so
    whatever its terms and sums lose shows a thousandfold in the draws.  Against 64 bits the streamed rows miss no more of 24576
    draws than the general routines' weights of 24 bits, summed in double, do: their number and four times its spread."""
    B, H, W, missed, general = 2, 64, 64, 0, 0
    for seed in (1, 2, 3):
        cfg = synth.RoundConfig("near", B=B, H=H, W=W, V=V, dtype=dtype, sigma=0.003, cfg_scale=0.0, top_k=top_k,
                                resample_mode=binding.RESAMPLE_RESIDUAL_ALL, seed=seed)
        batch = pu.build_batch(cfg)
        p = binding.params_from_config(cfg)
        ctx.ensure_workspace(p)
        tok_hi = torch.empty((B, H, W), dtype=torch.int32, device="cuda")
        stats, q_hi = torch.empty((B, cfg.h, cfg.w, 4), device="cuda"), torch.empty((B, H, W), device="cuda")
        everywhere = torch.full((B, H, 2), -1, dtype=torch.int32, device="cuda")
        want = torch.empty((B, H, W), dtype=torch.int64, device="cuda")

        def prob(z):
            e = torch.where(z >= torch.topk(z, top_k, dim=-1).values[..., -1:], torch.exp(z - z.amax(-1, keepdim=True)), 0.0)
            return e / e.sum(-1, keepdim=True)

        for b in range(B):
            u = torch.tensor([orc.position_uniforms(seed, b, t, cfg.round)[1] for t in range(H * W)], dtype=torch.float64, device="cuda")
            q = prob(batch["draft_lo"][b].double()).repeat_interleave(cfg.r, 0).repeat_interleave(cfg.r, 1)
            cdf = (prob(batch["cond"][b].double()) - q).clamp_min_(0.0).view(-1, V).cumsum(-1)
            want[b] = torch.searchsorted(cdf, (u * cdf[:, -1]).unsqueeze(-1), right=True).view(H, W)
        for how in (False, True):
            ctx.set_general_path_only(how)
            out = torch.empty((B, H, W), dtype=torch.int32, device="cuda")
            ctx.mulo_upsample_pool(p, batch["draft_lo"], batch["tok_lo"], None, tok_hi, stats, q_hi)
            n0 = ctx.kernel_launches()
            ctx.mulo_resample(p, batch["cond"], None, batch["draft_lo"], stats, tok_hi, None, everywhere, everywhere, out)
            if how:
                general += int((out.long() != want).sum())
            else:
                missed += int((out.long() != want).sum())
                assert ctx.kernel_launches() - n0 >= 2   # streamed
        ctx.set_general_path_only(False)
    assert missed <= general + 4 * np.sqrt(general + 1.0), (missed, general)


@pytest.mark.parametrize("V,top_k,dtype", [(16384, 2048, "bf16"), (8192, 1000, "f32"), (12296, 1537, "bf16")])
def test_sums_of_streamed_stages(ctx, V, top_k, dtype):
    """Z_q, p(x~) and q(x~) of the stages on more rows than are kept in shared memory, against 64 bits: a sum is no further off than
    that of the general routines (which the same bound holds for), the probabilities hardly more than their rounding to fp32, which
    makes a mean relative error of 0.36 * 2^-24."""
    cfg = dataclasses.replace(BASE, H=52, W=52, V=V, top_k=top_k, dtype=dtype, temperature=0.8 if dtype == "f32" else 1.0)
    batch = pu.build_batch(cfg)
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    n0 = ctx.kernel_launches()
    g = pu.gpu_stages(ctx, cfg, batch)
    assert ctx.kernel_launches() - n0 >= 2 + 3 + 1 + 2   # streamed, all of them
    ctx.set_general_path_only(True)
    general = pu.gpu_stages(ctx, cfg, batch)
    ctx.set_general_path_only(False)
    o = pu.oracle_images(cfg, batch, [0])[0]
    want = orc.upsample_pool_image(pu.orc_params(cfg, 0), synth.to_numpy_logits(batch["draft_lo"][0]), batch["tok_lo"][0].cpu().numpy())["stats"]
    e = {}
    for name, r in (("streamed", g), ("general", general)):
        z = r["stats"][0].astype(np.float64)
        e[name] = relative(z[..., 2] + z[..., 3], want[..., 2]).mean()
    assert e["streamed"] < 2.0 ** -26 and e["streamed"] <= 1.5 * e["general"], e
    for k in ("p_tok", "q_tok"):
        err, err_general = relative(g[k][0], o[k]).mean(), relative(general[k][0], o[k]).mean()
        assert err < 1.25 * 0.36 * 2.0 ** -24 and err <= 1.1 * err_general, (k, err, err_general)
