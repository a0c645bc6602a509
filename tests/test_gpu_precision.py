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
