"""GPU parity on rows with forbidden ids: logits at the lowest finite value of their type, in the conditional rows alone (guidance
then takes them to -inf) or in both.  Sums over such a row overflow, so that nothing may be derived from its mean or spread
without a check.  Everything against the CPU oracle, which sorts and exponentiates such rows like any others."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as orc
from paper_2601_05149_b200 import binding, synth

import parity_util as pu

pytestmark = pytest.mark.gpu

ROWS = synth.RoundConfig("forbidden", B=1, H=8, W=8, V=4096, dtype="bf16", sigma=1.0, top_k=500, radius=1, seed=801,
                         resample_mode=binding.RESAMPLE_ISOLATED_RESIDUAL)
EQ5 = dict(accept_mode=binding.ACCEPT_THRESHOLD, tau=1e-3, resample_mode=binding.RESAMPLE_TARGET_ALL)
NONE = dict(EQ5, tau=2.0)   # nothing is accepted
FEW = lambda cfg: 2
QUARTER = lambda cfg: cfg.V // 4
MOST = lambda cfg: cfg.V - cfg.top_k + 1   # the top_k-th largest value is a forbidden one


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    binding.lib()
    c = binding.Context(0)
    c.set_workspace(torch.empty(1 << 16, dtype=torch.uint8, device="cuda"))
    yield c
    c.close()


def forbid(cfg, n, both=False, block=False):
    """A batch whose rows all forbid the same n ids (`block`: consecutive ones); the guidance rows only if `both`."""
    batch = synth.build_batch(cfg, "cuda")
    ids = np.arange(8, 8 + n) if block else np.random.default_rng(cfg.seed).permutation(cfg.V)[:n]
    ids = torch.from_numpy(ids).cuda()
    low = torch.finfo(cfg.torch_dtype).min
    for k in ("cond", "draft_lo") + (("uncond",) if both and cfg.has_uncond else ()):
        batch[k][..., ids] = low
    pu.redraw_tokens(cfg, batch)
    return batch


FORMS = [dict(), dict(temperature=0.7), dict(cfg_scale=3.0), dict(cfg_scale=3.0, both=True), dict(dtype="f32", V=1032, top_k=129),
         dict(dtype="f32", V=1032, top_k=129, cfg_scale=3.0, temperature=0.9)]
form_id = lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "plain"


@pytest.mark.parametrize("how", ["stages", "general", "round"])
@pytest.mark.parametrize("n", [FEW, QUARTER, MOST], ids=["few", "quarter", "most"])
@pytest.mark.parametrize("form", FORMS, ids=form_id)
def test_rows_with_a_cut(ctx, form, n, how):
    form = dict(form)
    both = form.pop("both", False)
    cfg = dataclasses.replace(ROWS, **form)
    batch = forbid(cfg, n(cfg), both)
    ctx.set_general_path_only(how == "general")
    try:
        g = pu.gpu_stages(ctx, cfg, batch) if how == "stages" else pu.gpu_round(ctx, cfg, batch)
    finally:
        ctx.set_general_path_only(False)
    pu.check_round(cfg, g, pu.oracle_images(cfg, batch, [0]))
    assert ctx.poll_device_status() & ~binding.DEV_DENSE_FALLBACK == 0


@pytest.mark.parametrize("block", [False, True], ids=["scattered", "block"])
@pytest.mark.parametrize("n", [FEW, QUARTER, lambda cfg: cfg.V - 24], ids=["few", "quarter", "all-but-24"])
@pytest.mark.parametrize("cfg_scale", [0.0, 3.0])
@pytest.mark.parametrize("over", [
    dict(**EQ5), dict(pool_k=100, pool_delta=0.3, **EQ5), dict(V=4104, pool_k=100, pool_delta=0.3), dict(),
], ids=["flat", "full", "flat-pooled", "flat-residual"])
def test_rows_without_a_cut(ctx, over, cfg_scale, n, block):
    cfg = dataclasses.replace(ROWS, top_k=0, cfg_scale=cfg_scale, **over)
    batch = forbid(cfg, n(cfg), block=block)
    pu.check_round(cfg, pu.gpu_round(ctx, cfg, batch), pu.oracle_images(cfg, batch, [0]))
    assert ctx.poll_device_status() & ~binding.DEV_ZERO_DRAFT_PROB == 0


@pytest.mark.parametrize("n", [FEW, QUARTER, MOST], ids=["few", "quarter", "most"])
@pytest.mark.parametrize("V", [4096, 16392])   # the row in registers, in shared memory
@pytest.mark.parametrize("cfg_scale", [0.0, 3.0])
def test_redraw_and_draft_draws(ctx, cfg_scale, V, n):
    cfg = dataclasses.replace(ROWS, V=V, top_k=V // 8, cfg_scale=cfg_scale)
    batch = forbid(cfg, n(cfg))
    p = binding.params_from_config(cfg)
    ctx.ensure_workspace(p)
    for general in (False, True):
        tok = torch.full((1, cfg.h, cfg.w), -5, dtype=torch.int32, device="cuda")
        ctx.set_general_path_only(general)
        try:
            ctx.mulo_sample_draft(p, batch["draft_lo"], tok)
        finally:
            ctx.set_general_path_only(False)
        want, edge = orc.sample_draft_tokens(pu.orc_params(cfg, 0), synth.to_numpy_logits(batch["draft_lo"][0]), with_edge=True)
        assert not ((tok[0].cpu().numpy() != want) & (edge == 0)).any()

    steps = np.arange(1, 65, dtype=np.int32).reshape(8, 8) % 5   # four steps, and positions that stay
    out = torch.full((1, 8, 8), -7, dtype=torch.int32, device="cuda")
    pos = torch.empty(64, dtype=torch.int32, device="cuda")
    offsets = torch.empty(2 * 66, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_plan(p, torch.from_numpy(steps).cuda(), 64, pos, offsets)
    for s in range(1, 5):
        ctx.mulo_redraw_step(p, s, 64, pos, offsets, batch["cond"], batch["uncond"], out)
    cond = [synth.to_numpy_logits(batch["cond"][0])] * 4
    unc = [synth.to_numpy_logits(batch["uncond"][0])] * 4 if cfg.has_uncond else None
    want, _, edge = orc.redraw_loop(pu.orc_params(cfg, 0), steps, cond, unc, np.full((8, 8), -7, np.int32), with_edge=True)
    assert not ((out[0].cpu().numpy() != want) & (edge == 0)).any()


@pytest.mark.parametrize("over", [
    dict(top_k=0, **NONE), dict(top_k=0, pool_k=50, **NONE), dict(top_k=0, V=4104, pool_k=50, **NONE),
    dict(top_k=0, **{**NONE, "resample_mode": binding.RESAMPLE_RESIDUAL_ALL}), dict(top_k=0), dict(**NONE),
], ids=["flat", "full", "flat-pooled", "flat-residual", "flat-eq1", "rows"])
def test_rows_without_a_mass(ctx, over):
    """An id forbidden in the guidance rows alone mixes to +inf and no probability is a number: every draw says -1, and no
    token is what the workspace happened to hold."""
    cfg = dataclasses.replace(ROWS, cfg_scale=3.0, radius=0, **over)
    batch = pu.build_batch(cfg)
    batch["uncond"][..., 5] = torch.finfo(cfg.torch_dtype).min
    p = binding.params_from_config(cfg)
    ctx.set_workspace(torch.full((ctx.workspace_bytes(p),), 7, dtype=torch.uint8, device="cuda"))
    g = pu.gpu_round(ctx, cfg, batch)
    pu.check_round(cfg, g, pu.oracle_images(cfg, batch, [0]))
    if cfg.accept_mode == binding.ACCEPT_THRESHOLD:
        assert (g["reject"] == 1).all() and (g["out_tok"] == -1).all()


@pytest.mark.parametrize("V", [4096, 16392, 49160])
def test_draws_without_a_mass(ctx, V):
    cfg = dataclasses.replace(ROWS, V=V, top_k=V // 8, cfg_scale=3.0, temperature=0.7)
    batch = synth.build_batch(dataclasses.replace(cfg, H=4, W=4), "cuda")
    batch["uncond"][..., 5] = torch.finfo(cfg.torch_dtype).min
    batch["draft_lo"][..., 5] = torch.finfo(cfg.torch_dtype).max
    for top_k, general in ((0, False), (0, True), (cfg.top_k, False), (cfg.top_k, True)):
        p = binding.params_from_config(dataclasses.replace(cfg, H=4, W=4, top_k=top_k))
        ctx.ensure_workspace(p)
        tok = torch.full((1, 2, 2), 7, dtype=torch.int32, device="cuda")
        out = torch.full((1, 4, 4), 7, dtype=torch.int32, device="cuda")
        pos = torch.empty(16, dtype=torch.int32, device="cuda")
        offsets = torch.empty(2 * 18, dtype=torch.int32, device="cuda")
        ctx.set_general_path_only(general)
        try:
            ctx.mulo_sample_draft(p, batch["draft_lo"], tok)
        finally:
            ctx.set_general_path_only(False)
        ctx.mulo_redraw_plan(p, torch.ones((1, 4, 4), dtype=torch.int32, device="cuda"), 16, pos, offsets)
        ctx.mulo_redraw_step(p, 1, 16, pos, offsets, batch["cond"], batch["uncond"], out)
        assert (tok == -1).all() and (out == -1).all(), (top_k, general)
