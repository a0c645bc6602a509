"""GPU parity at the sizes where the row kernels change: smallest and largest rows, parts of a row that are empty or end
inside a piece, the lines between the kernels, neighbour lists that do not split evenly, rows that mislead a prediction.
Everything against the CPU oracle; the bound on probabilities and on excused positions is the one of parity_util."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2601_05149_b200 import binding, synth

import parity_util as pu
import test_gpu_redraw as redraw

pytestmark = pytest.mark.gpu

EQ5 = dict(accept_mode=binding.ACCEPT_THRESHOLD, tau=1e-3, resample_mode=binding.RESAMPLE_TARGET_ALL)
ALL = dict(resample_mode=binding.RESAMPLE_RESIDUAL_ALL)
FLAT = synth.RoundConfig("flat", B=2, H=6, W=4, V=16384, dtype="bf16", sigma=1.0, cfg_scale=3.0, top_k=0, radius=1, seed=501)
ROWS = synth.RoundConfig("rows", B=1, H=16, W=16, V=16384, dtype="bf16", sigma=1.0, cfg_scale=3.0, top_k=2000, radius=1, seed=601)


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    binding.lib()
    c = binding.Context(0)
    c.set_workspace(torch.empty(1 << 16, dtype=torch.uint8, device="cuda"))
    yield c
    c.close()


def parity(ctx, cfg, batch=None, kernel=None):
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    if kernel:
        assert ctx.round_kernel(p, cfg.has_uncond) == kernel
    batch = batch or pu.build_batch(cfg)
    g = pu.gpu_round(ctx, cfg, batch)
    pu.check_round(cfg, g, pu.oracle_images(cfg, batch, list(range(cfg.B))))
    assert ctx.poll_device_status() & ~(binding.DEV_DENSE_FALLBACK | binding.DEV_ZERO_DRAFT_PROB) == 0


@pytest.mark.parametrize("over", [
    dict(V=8, **EQ5), dict(V=8, **ALL),                                      # one lane has ids
    dict(V=520, dtype="f32", **EQ5), dict(V=520, dtype="f32", **ALL),       # groups without ids
    dict(V=4096, **EQ5), dict(V=4104, **EQ5),                                # four whole pieces per thread, and one id more
    dict(V=16384, **ALL), dict(V=16392, **ALL), dict(V=16376, temperature=0.9, **ALL),
    dict(V=16384, temperature=0.9, **EQ5), dict(V=16384, temperature=0.9, **ALL), dict(V=4096, dtype="f32", temperature=1.3, **ALL),   # even, scaled
    dict(V=8192, temperature=0.9, pool_k=300, pool_delta=0.2),
    dict(V=65536, H=2, **EQ5), dict(V=65536, H=2, dtype="f32", cfg_scale=0.0, **EQ5),
    dict(V=56320, H=2, **ALL), dict(V=65528, H=2, **ALL),                    # the largest weights in shared memory; too large for it
    dict(V=2048, H=16, W=16, r=8, **ALL),                                    # 64 rows under a draft row
    dict(V=4096, pool_k=2, pool_delta=0.3), dict(V=4096, pool_k=2048, pool_delta=0.9), dict(V=4096, pool_k=2047, pool_delta=0.9),
    dict(V=12296, pool_k=257, pool_delta=0.2, **EQ5), dict(V=8192, dtype="f32", pool_k=1000, pool_delta=0.0),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()))
def test_rows_without_a_cut(ctx, over):
    cfg = dataclasses.replace(FLAT, **over)
    parity(ctx, cfg, kernel="general" if cfg.V == 65528 else "full")


@pytest.mark.parametrize("V,cfg_scale,kernel", [(57344, 0.0, "full"), (65536, 0.0, "full"), (65528, 0.0, "general"), (65536, 3.0, "general")])
def test_pooled_rows_of_large_vocabularies(ctx, V, cfg_scale, kernel):
    """Weights of so many ids do not fit in shared memory, a raw bf16 row without guidance does."""
    cfg = dataclasses.replace(FLAT, V=V, H=2, cfg_scale=cfg_scale, pool_k=64, pool_delta=0.2, **EQ5)
    parity(ctx, cfg, kernel=kernel)


@pytest.mark.parametrize("r,H,W", [(5, 20, 35), (8, 16, 32), (9, 18, 27), (16, 32, 16), (12, 12, 12)])
@pytest.mark.parametrize("over,kernel", [(dict(top_k=300), "lane"), (dict(top_k=300, pool_k=40, pool_delta=0.3), "stream")], ids=["plain", "pooled"])
def test_many_rows_with_a_cut_under_a_draft_row(ctx, over, kernel, r, H, W):
    """More children than the sixteen whose uniforms are kept at a time, and parents split over thread blocks."""
    parity(ctx, dataclasses.replace(ROWS, H=H, W=W, r=r, V=2048, **over), kernel=kernel)


@pytest.mark.parametrize("over", [dict(), EQ5, ALL, dict(pool_k=40, pool_delta=0.3, **EQ5)], ids=["mixed", "eq5", "residual", "pooled-eq5"])
def test_rows_without_a_cut_at_large_ratios(ctx, over):
    """Beyond k_round_flat's ratio: the general routines."""
    pooled_target = over.get("pool_k", 1) > 1   # k_round_full's, whatever the ratio
    cfg = dataclasses.replace(ROWS, H=24, W=12, r=12, V=2048, top_k=0, **over)
    parity(ctx, cfg, kernel="full" if pooled_target else "general")


def test_rows_without_a_cut_that_mislead_the_prediction(ctx):
    """Consecutive rows whose maxima lie tens apart (every other one is streamed again), constant rows, and one-hot ones."""
    for over in (EQ5, ALL, dict(pool_k=300, pool_delta=0.2)):
        cfg = dataclasses.replace(FLAT, V=4104, cfg_scale=0.0, **over)
        batch = pu.build_batch(cfg)
        x = batch["cond"].view(-1, cfg.V)
        x[0::4] += 60.0
        x[1::4] -= 35.0
        x[2] = 1.5
        x[3] = -30.0
        x[3, 7] = 30.0
        batch["draft_lo"].view(-1, cfg.V)[1::2] += 50.0
        pu.redraw_tokens(cfg, batch)
        parity(ctx, cfg, batch, "full")


@pytest.mark.parametrize("over,kernel", [
    (dict(B=5, H=27, W=34, V=4096, top_k=512, r=1), "lane"),   # one row under each draft row, several of them per thread block
    (dict(V=1024, top_k=16), "lane"), (dict(V=1032, top_k=128), "lane"),
    (dict(V=2056, top_k=257, dtype="f32", cfg_scale=0.0, temperature=0.9), "lane"),
    (dict(V=16384, top_k=3276), "lane"), (dict(V=4096, top_k=1024), "lane"), (dict(V=4096, top_k=1200), "lane"),   # two warps, four
    (dict(V=16384, top_k=2048, dtype="f32"), "lane"), (dict(V=16384, top_k=1024, dtype="f32"), "lane"),   # four again, for their lists' bytes; two
    (dict(V=16384, top_k=2048, dtype="f32", pool_k=300, pool_delta=0.3), "stream"),
    (dict(V=49152, top_k=6144, H=4, W=8), "stream"), (dict(V=4096, top_k=1900), "general"),   # lists too long for it; half of the row
    (dict(V=8192, top_k=1000, pool_k=500, pool_delta=0.3), "stream"), (dict(V=8192, top_k=1000, pool_k=513, pool_delta=0.9), "stream"),
    (dict(V=4104, top_k=500, pool_k=2048, pool_delta=0.05, dtype="f32", radius=2, resample_mode=binding.RESAMPLE_ISOLATED_RESIDUAL),
     "stream"),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) if isinstance(o, dict) else o)
def test_rows_with_a_cut(ctx, over, kernel):
    cfg = dataclasses.replace(ROWS, **over)
    ctx.poll_fallback_counts()
    parity(ctx, cfg, kernel=kernel)
    # (the kernel did its rows itself: what it hands to the general routines is the exception)
    assert ctx.poll_fallback_counts()[0] <= cfg.B * cfg.H * cfg.W // 20


@pytest.mark.parametrize("W", [37, 38], ids=["few", "many"])   # 592 and 608 draft rows: four per SM, and more
@pytest.mark.parametrize("V,dtype", [(264, "bf16"), (8192, "f32"), (16392, "bf16")])
def test_draft_sums_without_a_cut(ctx, V, dtype, W):
    """Sums in double of fp32 weights of 2^-22 each, as an fp32 pair; q(x~) is rounded to fp32 besides."""
    cfg = dataclasses.replace(FLAT, B=1, H=16, W=W, r=1, V=V, dtype=dtype, temperature=0.9)
    batch = pu.build_batch(cfg)
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    hi, q = torch.empty((1, 16, W), dtype=torch.int32, device="cuda"), torch.empty((1, 16, W), device="cuda")
    stats = torch.empty((1, 16, W, 4), device="cuda")
    ctx.mulo_upsample_pool(p, batch["draft_lo"], batch["tok_lo"], None, hi, stats, q)
    tok = batch["tok_lo"][0].cpu().numpy()
    want = orc.upsample_pool_image(pu.orc_params(cfg, 0), synth.to_numpy_logits(batch["draft_lo"][0]), tok)
    got = stats[0].double().cpu().numpy()
    assert np.array_equal(hi[0].cpu().numpy(), tok) and np.array_equal(got[..., 0], want["stats"][..., 0])
    assert np.array_equal(got[..., 1], want["stats"][..., 1])
    np.testing.assert_allclose(got[..., 2] + got[..., 3], want["stats"][..., 2], rtol=2.0 ** -22)
    np.testing.assert_allclose(q[0].cpu().numpy(), want["q_tok"], rtol=2.0 ** -22 + 2.0 ** -24)


@pytest.mark.parametrize("V", [16384, 16392, 49152, 49160])
@pytest.mark.parametrize("how", ["none", "ties", "const"])
def test_general_path_around_shared_memory(ctx, V, how):
    """Rows in registers, in shared memory and beyond it, with masses of ties at the threshold."""
    cfg = dataclasses.replace(ROWS, H=4, W=4, V=V, top_k=V // 8, cfg_scale=0.0 if how == "const" else 3.0, seed=701, **ALL)
    batch = pu.build_batch(cfg)
    for k in ("cond", "uncond", "draft_lo"):
        if batch[k] is not None and how != "none":
            x = torch.round(batch[k].float()) if how == "ties" else torch.zeros_like(batch[k].float())
            batch[k] = x.to(batch[k].dtype).contiguous()
    pu.redraw_tokens(cfg, batch)
    ctx.set_general_path_only(True)
    try:
        parity(ctx, cfg, batch, "general")
    finally:
        ctx.set_general_path_only(False)


@pytest.mark.parametrize("V", [16384, 16392, 49152, 65536])
def test_redraw_around_shared_memory(ctx, V):
    redraw.test_redraw_steps_against_oracle(ctx, dict(B=1, H=4, W=12, V=V, dtype="bf16", top_k=V // 8, cfg_scale=2.0,
                                                      temperature=0.9, window=4, density=0.5))


STAGES = synth.RoundConfig("stages", B=4, H=24, W=26, V=4096, dtype="bf16", sigma=1.0, cfg_scale=3.0, top_k=500, radius=1, seed=1201)


@pytest.mark.parametrize("over", [
    dict(), dict(V=1024, top_k=100, dtype="f32"), dict(V=4104, top_k=600, cfg_scale=0.0, temperature=0.8), dict(V=16384, top_k=2000),
    dict(V=8192, top_k=2600), dict(r=1, H=20, W=31, V=8192, sigma=0.1, cfg_scale=0.0, radius=0), dict(r=3, H=24, W=27, radius=2, sigma=0.3), dict(B=2, H=36, W=36, resample_mode=binding.RESAMPLE_RESIDUAL_ALL),
    dict(resample_mode=binding.RESAMPLE_TARGET_ALL), dict(accept_mode=binding.ACCEPT_THRESHOLD, tau=1e-3),
    dict(resample_mode=binding.RESAMPLE_ISOLATED_RESIDUAL, radius=3), dict(cubed=True), dict(quantum=0.5, cfg_scale=0.0),
    dict(r=1, H=20, W=31, V=8192, top_k=1000, quantum=0.5), dict(shift=True),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "plain")
def test_stages_of_many_rows(ctx, over):
    """More rows than the stages keep in shared memory: the streaming kernels, rows that mislead their predictions included."""
    over = dict(over)
    cubed, quantum, shift = over.pop("cubed", False), over.pop("quantum", 0.0), over.pop("shift", False)
    cfg = dataclasses.replace(STAGES, **over)
    batch = pu.build_batch(cfg)
    for k in ("cond", "uncond", "draft_lo"):
        if batch[k] is None:
            continue
        if cubed:
            batch[k] = (batch[k].float() ** 3 / 8).to(batch[k].dtype)
        if quantum:
            batch[k] = ((batch[k].float() / quantum).round() * quantum).to(batch[k].dtype)
        if shift:     # every other row lies 20 higher
            batch[k][:, :, ::2] += 20.0
    pu.redraw_tokens(cfg, batch)
    n0 = ctx.kernel_launches()
    g = pu.gpu_stages(ctx, cfg, batch)
    isolated = cfg.resample_mode == binding.RESAMPLE_ISOLATED_RESIDUAL
    few = cfg.B * cfg.h * cfg.w <= (4 if cfg.V > 4096 else 16) * torch.cuda.get_device_properties(0).multi_processor_count
    assert ctx.kernel_launches() - n0 == (1 if few else 2) + 3 + 1 + (1 if isolated else 2)   # the fast paths, but for few draft rows
    o = pu.oracle_images(cfg, batch, list(range(cfg.B)))
    pu.check_round(cfg, g, o)
    for b in range(cfg.B):
        want = orc.upsample_pool_image(pu.orc_params(cfg, b), synth.to_numpy_logits(batch["draft_lo"][b]), batch["tok_lo"][b].cpu().numpy())
        np.testing.assert_array_equal(g["tok_hi"][b], want["tok_hi"])
        np.testing.assert_allclose(g["stats"][b].astype(np.float64)[..., 0:2], want["stats"][..., 0:2], rtol=0, atol=0)
        np.testing.assert_allclose(g["stats"][b][..., 2].astype(np.float64) + g["stats"][b][..., 3], want["stats"][..., 2], rtol=1e-6)
    assert ctx.poll_device_status() & ~(binding.DEV_DENSE_FALLBACK | binding.DEV_ZERO_DRAFT_PROB) == 0


@pytest.mark.parametrize("over", [dict(), dict(r=3, H=24, W=27), dict(V=8192, top_k=1000, dtype="f32", cfg_scale=0.0), dict(V=8192, top_k=900)],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "plain")
@pytest.mark.parametrize("tied", ["target", "draft"])
def test_rows_that_the_stages_leave(ctx, tied, over):
    """Rows with hundreds of equal logits at the threshold crowd a bin (target rows, the draft rows' statistics) or overflow the list
    of what lies above a given threshold (draft rows of the redraw, with all rows under them): each stage has to leave some to
    the general routines, and says so."""
    cfg = dataclasses.replace(STAGES, resample_mode=binding.RESAMPLE_RESIDUAL_ALL, **over)
    batch = pu.build_batch(cfg)
    for k in ("cond", "uncond") if tied == "target" else ("draft_lo",):
        if batch[k] is not None:
            batch[k] = ((batch[k].float() / 2.0).round() * 2.0).to(batch[k].dtype)
    pu.redraw_tokens(cfg, batch)
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    B, H, W = cfg.B, cfg.H, cfg.W
    o = binding.alloc_round_outputs(p, "cuda")
    tok_hi = torch.empty((B, H, W), dtype=torch.int32, device="cuda")
    stats, q_hi = torch.empty((B, cfg.h, cfg.w, 4), device="cuda"), torch.empty((B, H, W), device="cuda")

    def left():
        torch.cuda.synchronize()
        assert ctx.poll_device_status() & ~(binding.DEV_DENSE_FALLBACK | binding.DEV_ZERO_DRAFT_PROB) == 0
        return ctx.poll_fallback_counts()[0]

    left()
    n0 = ctx.kernel_launches()
    ctx.mulo_upsample_pool(p, batch["draft_lo"], batch["tok_lo"], None, tok_hi, stats, q_hi)
    assert (left() > 0) == (tied == "draft" and ctx.kernel_launches() - n0 == 2)   # (few draft rows are not streamed)
    ctx.mulo_verify(p, batch["cond"], batch["uncond"], batch["draft_lo"], stats, tok_hi, None, o["p_tok"], o["q_tok"], o["accept_prob"],
                    o["reject_bits"], o["n_reject"], o["first_reject"])
    assert (left() > 0) == (tied == "target")
    ctx.mulo_local_reject_expand(p, o["reject_bits"], o["first_reject"], o["expand_bits"], o["n_expand"])
    ctx.mulo_resample(p, batch["cond"], batch["uncond"], batch["draft_lo"], stats, tok_hi, None, o["reject_bits"], o["expand_bits"],
                      o["out_tok"])
    assert left() > 0
    pu.check_round(cfg, pu.finish_outputs(o, W), pu.oracle_images(cfg, batch, list(range(B))))


@pytest.mark.parametrize("over", [dict(), dict(B=3, H=30, W=37, r=1, V=1024, top_k=100), dict(B=5, H=48, W=45, r=3, radius=2),
                                  dict(B=5, H=3, W=1500, r=3, V=1024, top_k=100)],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "plain")
@pytest.mark.parametrize("density", [0.0, 0.0005, 0.02, 0.5, 1.0, "ends"])
def test_redraw_of_any_share_of_the_grid(ctx, over, density):
    """The streamed redraw finds the positions of R_X by itself: none, one or two, some, all; bits past a row's end count as nothing.  "ends": all of the
    first and of the last image, nothing between."""
    cfg = dataclasses.replace(STAGES, resample_mode=binding.RESAMPLE_MIXED, **over)
    batch = pu.build_batch(cfg)
    pu.redraw_tokens(cfg, batch)
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    B, H, W = cfg.B, cfg.H, cfg.W
    g = torch.Generator(device="cuda").manual_seed(77)
    hits = torch.rand((B, H, (W + 31) // 32, 32), generator=g, device="cuda") < (1.0 if density == "ends" else density)
    if density == "ends":
        hits[1:B - 1] = False
    if density == 0.0005:
        hits.view(-1)[:] = False
        hits[B - 1, H - 1, (W - 1) // 32, (W - 1) % 32] = True
        hits[0, 1, 0, 2] = True
    also = torch.rand(hits.shape, generator=g, device="cuda") < 0.5
    past = torch.arange(hits.shape[2] * 32, device="cuda").view(1, 1, -1, 32) >= W

    def words(bits):
        w = (bits.to(torch.int64) << torch.arange(32, device="cuda")).sum(-1)
        return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32).contiguous()

    expand, reject = words(hits | past), words(hits & also)
    tok_hi = torch.empty((B, H, W), dtype=torch.int32, device="cuda")
    stats, q_hi = torch.empty((B, cfg.h, cfg.w, 4), device="cuda"), torch.empty((B, H, W), device="cuda")
    ctx.mulo_upsample_pool(p, batch["draft_lo"], batch["tok_lo"], None, tok_hi, stats, q_hi)
    out = {}
    for how in (False, True):
        out[how] = torch.full((B, H, W), -9, dtype=torch.int32, device="cuda")
        ctx.set_general_path_only(how)
        n0 = ctx.kernel_launches()
        ctx.mulo_resample(p, batch["cond"], batch["uncond"], batch["draft_lo"], stats, tok_hi, None, reject, expand, out[how])
        ctx.set_general_path_only(False)
        assert ctx.kernel_launches() - n0 == (1 if how else 2)
    inside = (hits & ~past).flatten(2)[..., :W]
    assert torch.equal(out[False][~inside], tok_hi[~inside])
    assert int((out[False] != out[True]).sum()) <= 1   # (another order of summation: a draw in 10^4 or fewer)


def test_redraws_on_two_streams_of_one_context(ctx):
    """mulo_resample keeps nothing in the workspace but status bits: two of them at a time on one context."""
    cfgs = [dataclasses.replace(STAGES, seed=s, resample_mode=m) for s, m in ((1301, binding.RESAMPLE_RESIDUAL_ALL), (1302, binding.RESAMPLE_MIXED))]
    jobs = []
    for cfg in cfgs:
        batch = pu.build_batch(cfg)
        pu.redraw_tokens(cfg, batch)
        g = pu.gpu_stages(ctx, cfg, batch)
        jobs.append((cfg, binding.params_from_config(cfg), batch, {k: torch.from_numpy(g[k]).cuda() for k in ("tok_hi", "stats", "reject_bits", "expand_bits")},
                     torch.from_numpy(g["out_tok"]).cuda()))
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    for _ in range(20):
        outs = [torch.full_like(j[4], -9) for j in jobs]
        torch.cuda.synchronize()
        for (cfg, p, batch, s, _), out, st in zip(jobs, outs, streams):
            ctx.mulo_resample(p, batch["cond"], batch["uncond"], batch["draft_lo"], s["stats"], s["tok_hi"], None, s["reject_bits"],
                              s["expand_bits"], out, stream=st)
        torch.cuda.synchronize()
        for j, out in zip(jobs, outs):
            assert torch.equal(out, j[4])
