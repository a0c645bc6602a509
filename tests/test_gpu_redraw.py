"""GPU parity of the step-by-step redraw of R_X (Sec. 3.4): the device-side plan (positions sorted by
schedule step) and one launch per step, against the oracle's redraw loop on the same per-step logits."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2601_05149_b200 import binding, synth

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available()
    binding.lib()
    c = binding.Context(0)
    yield c
    c.close()


def _schedule(rng, B, H, W, window, density):
    """R_X masks, their islands and schedule by the ORACLE (the device gets them as inputs)."""
    steps = np.zeros((B, H, W), np.int32)
    for b in range(B):
        seeds = rng.random((H, W)) < density
        rx, _ = orc.expand(seeds.astype(np.uint8), 1, 0)
        labels, _, _, _ = orc.islands(rx)
        steps[b], _ = orc.island_schedule(labels, window)
    return steps


@pytest.mark.parametrize("case", [
    dict(B=2, H=12, W=16, V=512, dtype="bf16", top_k=64, cfg_scale=2.0, temperature=1.0, window=16, density=0.04),
    dict(B=3, H=8, W=8, V=256, dtype="f32", top_k=0, cfg_scale=0.0, temperature=0.7, window=2, density=0.10),
    dict(B=1, H=6, W=40, V=1032, dtype="bf16", top_k=100, cfg_scale=0.0, temperature=1.0, window=4, density=0.5),
], ids=lambda c: f"{c['dtype']}-V{c['V']}-{c['B']}x{c['H']}x{c['W']}-w{c['window']}")
def test_redraw_steps_against_oracle(ctx, case):
    B, H, W, V = case["B"], case["H"], case["W"], case["V"]
    rng = np.random.default_rng(41)
    cfg = synth.RoundConfig("redraw", B=B, H=H, W=W, V=V, r=1, dtype=case["dtype"], top_k=case["top_k"],
                            cfg_scale=case["cfg_scale"], temperature=case["temperature"], seed=4242, round=2)
    steps = _schedule(rng, B, H, W, case["window"], case["density"])
    n_steps = int(steps.max())
    assert n_steps >= 3
    g = torch.Generator(device="cuda").manual_seed(99)
    dt = cfg.torch_dtype
    cond = [(2.0 * torch.randn((B, H, W, V), generator=g, device="cuda")).to(dt) for _ in range(n_steps)]
    unc = [(c.float() + torch.randn((B, H, W, V), generator=g, device="cuda")).to(dt) for c in cond] \
        if cfg.has_uncond else None
    start = torch.from_numpy(rng.integers(0, V, (B, H, W)).astype(np.int32)).cuda()

    p = binding.params_from_config(cfg, image_offset=3)
    max_step = H * W                       # the bound a caller has without reading n_steps back
    guard = pu.Guarded("cuda")
    pos_list = guard.empty("pos_list", (B * H * W,), torch.int32)
    offsets = guard.empty("step_offsets", (2 * (max_step + 2),), torch.int32)
    out = guard.empty("out_tok", (B, H, W), torch.int32)
    out.copy_(start)
    d_steps = torch.from_numpy(steps).cuda()
    n0 = ctx.kernel_launches()
    ctx.mulo_redraw_plan(p, d_steps, max_step, pos_list, offsets)
    for s in range(1, n_steps + 1):
        ctx.mulo_redraw_step(p, s, max_step, pos_list, offsets, cond[s - 1], None if unc is None else unc[s - 1], out)
    torch.cuda.synchronize()
    guard.check()
    assert ctx.kernel_launches() - n0 == 3 + n_steps         # one launch per sequential step

    # the plan: slice s of the list holds exactly the positions of step s
    off = offsets.cpu().numpy()
    lst = pos_list.cpu().numpy()
    flat = steps.ravel()
    for s in range(1, n_steps + 1):
        assert sorted(lst[off[s]:off[s + 1]].tolist()) == np.flatnonzero(flat == s).tolist()
    assert off[n_steps + 1] == (flat > 0).sum() == off[max_step + 1]

    got = out.cpu().numpy()
    differ = flagged = 0
    for b in range(B):
        want, calls, edge = orc.redraw_loop(
            pu.orc_params(cfg, b + 3), steps[b], [synth.to_numpy_logits(c[b]) for c in cond],
            None if unc is None else [synth.to_numpy_logits(u[b]) for u in unc], start[b].cpu().numpy(), with_edge=True)
        assert calls == int(steps[b].max())
        bad = got[b] != want
        assert not (bad & (edge == 0)).any(), np.argwhere(bad & (edge == 0))[:5]
        assert np.array_equal(got[b][steps[b] == 0], start[b].cpu().numpy()[steps[b] == 0])
        differ += int(bad.sum())
        flagged += int(edge.sum())
    n_rx = int((steps > 0).sum())
    print(f"[redraw] {n_rx} positions over {n_steps} steps, flagged {flagged}, differing {differ}")
    assert differ <= max(1, int(1e-3 * n_rx))


def test_redraw_arguments_are_checked(ctx):
    p = binding.make_params(1, 8, 8, 256, 1, binding.F32)
    t = torch.zeros(64, dtype=torch.int32, device="cuda")
    off = torch.zeros(2 * 66, dtype=torch.int32, device="cuda")
    with pytest.raises(binding.MuloError) as e:
        ctx.mulo_redraw_plan(p, t, 0, t, off)
    assert e.value.status == binding.ERR_INVALID_ARG
    with pytest.raises(binding.MuloError) as e:
        ctx.mulo_redraw_plan(p, t, 65, t, off)             # more steps than positions
    assert e.value.status == binding.ERR_INVALID_ARG
    logits = torch.zeros((1, 8, 8, 256), device="cuda")
    for s in (0, 65):
        with pytest.raises(binding.MuloError) as e:
            ctx.mulo_redraw_step(p, s, 64, t, off, logits, None, t)
        assert e.value.status == binding.ERR_INVALID_ARG


@pytest.mark.parametrize("V", [512, 16392, 49160])   # the row in registers, in shared memory, beyond it
@pytest.mark.parametrize("captured", [False, True], ids=["stream", "graph"])
def test_logits_and_plan_are_rewritten_between_steps(ctx, captured, V):
    """What a host with a model does: one logits buffer that every step's model call writes anew, one pair of plan buffers that the
    next round's plan overwrites while the last steps may still run -- on one stream without a wait, and as one graph.  Steps are
    launched ahead of their predecessors' end, so each must see what was written just before it."""
    B, H, W = 2, 6, 10
    rng = np.random.default_rng(V)
    cfg = synth.RoundConfig("rewritten", B=B, H=H, W=W, V=V, r=1, dtype="bf16", top_k=V // 8, cfg_scale=2.0, seed=77, round=1)
    plans = [_schedule(rng, B, H, W, 3, density) for density in (0.10, 0.25)]
    n_steps = [int(s.max()) for s in plans]
    g = torch.Generator(device="cuda").manual_seed(V)
    cond = [(2.0 * torch.randn((B, H, W, V), generator=g, device="cuda")).bfloat16() for _ in range(sum(n_steps))]
    unc = [(c.float() + torch.randn((B, H, W, V), generator=g, device="cuda")).bfloat16() for c in cond]
    start = torch.from_numpy(rng.integers(0, V, (B, H, W)).astype(np.int32)).cuda()
    d_plans = [torch.from_numpy(s).cuda() for s in plans]
    p = binding.params_from_config(cfg)
    buf_c, buf_u = torch.empty_like(cond[0]), torch.empty_like(cond[0])
    pos_list = torch.empty(B * H * W, dtype=torch.int32, device="cuda")
    offsets = torch.empty(2 * (H * W + 2), dtype=torch.int32, device="cuda")
    out = torch.empty_like(start)

    def rounds():
        out.copy_(start)
        at = 0
        for d_step, n in zip(d_plans, n_steps):
            ctx.mulo_redraw_plan(p, d_step, H * W, pos_list, offsets)
            for s in range(1, n + 1):
                buf_c.copy_(cond[at])
                buf_u.copy_(unc[at])
                at += 1
                ctx.mulo_redraw_step(p, s, H * W, pos_list, offsets, buf_c, buf_u, out)

    if captured:
        rounds()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            rounds()
        for t in (buf_c, buf_u, pos_list, offsets, out):
            t.zero_()
        graph.replay()
        graph.replay()
    else:
        rounds()
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for b in range(B):
        tok, edge, at = start[b].cpu().numpy(), np.zeros((H, W), bool), 0
        for steps, n in zip(plans, n_steps):
            tok, _, e = orc.redraw_loop(pu.orc_params(cfg, b), steps[b], [synth.to_numpy_logits(c[b]) for c in cond[at:at + n]],
                                        [synth.to_numpy_logits(u[b]) for u in unc[at:at + n]], tok, with_edge=True)
            edge |= e != 0
            at += n
        bad = got[b] != tok
        assert not (bad & ~edge).any(), np.argwhere(bad & ~edge)[:5]
        assert bad.sum() <= 1


def test_a_step_of_more_positions_than_thread_blocks(ctx):
    B, H, W, V = 3, 16, 24, 264
    cfg = synth.RoundConfig("many", B=B, H=H, W=W, V=V, r=1, dtype="f32", top_k=40, cfg_scale=0.0, seed=78)
    cond = synth.build_batch(cfg, "cuda")["cond"]
    steps = np.ones((B, H, W), np.int32)
    p = binding.params_from_config(cfg)
    pos_list = torch.empty(B * H * W, dtype=torch.int32, device="cuda")
    offsets = torch.empty(2 * 3, dtype=torch.int32, device="cuda")
    out = torch.full((B, H, W), -7, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_plan(p, torch.from_numpy(steps).cuda(), 1, pos_list, offsets)
    ctx.mulo_redraw_step(p, 1, 1, pos_list, offsets, cond, None, out)
    for b in range(B):
        want, _, edge = orc.redraw_loop(pu.orc_params(cfg, b), steps[b], [synth.to_numpy_logits(cond[b])], None,
                                        np.zeros((H, W), np.int32), with_edge=True)
        assert not ((out[b].cpu().numpy() != want) & (edge == 0)).any()


def test_one_context_from_several_threads():
    """Calls that need no workspace, from four threads on one new context, each on its own stream and over its own sizes (every one
    asks for its kernels' limits anew): the tokens and steps are those of one thread."""
    import concurrent.futures as cf
    rng = np.random.default_rng(5)
    jobs = []
    for k in range(4):
        per = []
        for V in (256 + 1024 * k, 4104 + 4096 * k, 20000 + 4000 * k):
            H, W = 6 + k, 9
            labels = torch.from_numpy(orc.islands((rng.random((H, W)) < 0.5).astype(np.uint8))[0][None]).cuda()
            cfg = synth.RoundConfig("threads", B=1, H=H, W=W, V=V, r=1, dtype="bf16", top_k=V // 8, seed=k)
            per.append((cfg, labels, synth.build_batch(cfg, "cuda")["cond"]))
        jobs.append(per)

    def work(ctx, per, stream):
        res = []
        with torch.cuda.stream(stream):
            for cfg, labels, cond in per:
                p = binding.params_from_config(cfg)
                n = cfg.H * cfg.W
                step, out = torch.empty_like(labels), torch.zeros_like(labels)
                n_steps = torch.empty(1, dtype=torch.int32, device="cuda")
                pos, off = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(2 * (n + 2), dtype=torch.int32, device="cuda")
                ctx.mulo_island_schedule(p, labels, 3, step, n_steps)
                ctx.mulo_redraw_plan(p, step, n, pos, off)
                for s in range(1, 9):
                    ctx.mulo_redraw_step(p, s, n, pos, off, cond, None, out)
                res += [step.cpu().numpy(), out.cpu().numpy()]
        return res

    torch.cuda.synchronize()
    alone = binding.Context(0)
    want = [work(alone, per, torch.cuda.Stream()) for per in jobs]
    shared = binding.Context(0)
    with cf.ThreadPoolExecutor(4) as ex:
        got = list(ex.map(lambda per: work(shared, per, torch.cuda.Stream()), jobs))
    for a, b in zip(want, got):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)
    alone.close()
    shared.close()


_EARLY_WRITER = r"""
extern "C" __global__ void early_writer(const uint4* src, uint4* dst, long long n, const int* new_list, int* list, int n_list) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // what comes after may begin now, and is to find the old contents: 60 us and no more
  const long long t0 = clock64();
  while (clock64() - t0 < 120000) {}
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) dst[i] = src[i];
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < n_list; i += blockDim.x) list[i] = new_list[i];
}
"""


@pytest.mark.parametrize("V", [520, 8192, 16384, 20000, 49160])   # one, two, four pieces per thread; two and four CTAs to a row
@pytest.mark.parametrize("what", ["logits", "one id", "list", "nothing"])
def test_a_row_drawn_ahead_of_its_inputs(ctx, V, what):
    """The kernel before the step lets it begin and only then rewrites the row's logits (all of them, or one id of each row's last
    pieces) or the list: the step's token is that of what stands there when that kernel is done."""
    B, H, W = 2, 4, 16
    cfg = synth.RoundConfig("ahead", B=B, H=H, W=W, V=V, r=1, dtype="bf16", top_k=V // 8, cfg_scale=0.0, seed=79)
    p = binding.params_from_config(cfg)
    g = torch.Generator(device="cuda").manual_seed(V)
    old = (2.0 * torch.randn((B, H, W, V), generator=g, device="cuda")).bfloat16()
    new = old.clone()
    if what == "logits":
        new.copy_(2.0 * torch.randn((B, H, W, V), generator=g, device="cuda"))
    elif what == "one id":
        new[..., V - 3] = 40.0       # takes the whole mass
    steps = torch.zeros((B, H, W), dtype=torch.int32, device="cuda")
    steps.view(-1)[::17] = 1
    n = B * H * W
    pos, off = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(2 * 3, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_plan(p, steps, 1, pos, off)
    listed = pos.clone()
    if what == "list":
        listed[:8] = (listed[:8] + 5) % n
    want = torch.full((B, H, W), -7, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_step(p, 1, 1, listed, off, new, None, want)
    torch.cuda.synchronize()
    kernel = torch.cuda._compile_kernel(_EARLY_WRITER, "early_writer", compute_capability="100a")
    for _ in range(3):
        buf, lst = old.clone(), pos.clone()
        out = torch.full_like(want, -7)
        torch.cuda.synchronize()
        kernel(grid=(16, 1, 1), block=(256, 1, 1), args=[new, buf, buf.numel() // 8, listed, lst, 8])
        ctx.mulo_redraw_step(p, 1, 1, lst, off, buf, None, out)
        assert torch.equal(out, want)


def _shifted(pos, off):
    """The plan with position 1 in step 1."""
    off = off.clone()
    off[2:4] += 1
    return torch.cat([torch.tensor([1], dtype=torch.int32, device="cuda"), pos[:-1]]).contiguous(), off


_LATE_LISTS = r"""
extern "C" __global__ void late_lists(const int* new_off, int* off, int n_off, const int* new_list, int* list, int n_list, int cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
  for (int i = threadIdx.x; i < n_list; i += blockDim.x) list[i] = new_list[i];
  for (int i = threadIdx.x; i < n_off; i += blockDim.x) off[i] = new_off[i];
}
"""


@pytest.mark.parametrize("V", [520, 8192, 16384, 20000, 49160])   # one, two and four CTAs to a row
@pytest.mark.parametrize("more", [0, 90])
def test_a_list_rewritten_while_the_step_begins(ctx, V, more):
    """The kernel before the step lets it begin and rewrites offsets and list at any moment of the step's first 10 us: the step before
    gains a position, so both shift by one and an entry may be seen with either offset; or the step itself gains 90, more than it has
    clusters.  What counts is what stands there in the end."""
    B, H, W = 2, 4, 16
    cfg = synth.RoundConfig("late", B=B, H=H, W=W, V=V, r=1, dtype="bf16", top_k=V // 8, cfg_scale=0.0, seed=81)
    p = binding.params_from_config(cfg)
    g = torch.Generator(device="cuda").manual_seed(V)
    z = (2.0 * torch.randn((B, H, W, V), generator=g, device="cuda")).bfloat16()
    n = B * H * W

    def plan(steps):
        pos, off = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(2 * 4, dtype=torch.int32, device="cuda")
        ctx.mulo_redraw_plan(p, steps, 2, pos, off)
        return pos, off

    steps = torch.zeros((B, H, W), dtype=torch.int32, device="cuda")
    steps.view(-1)[3:24:3] = 2
    pos0, off0 = plan(steps)
    if more:
        steps.view(-1)[24:24 + more] = 2
        pos1, off1 = plan(steps)
    else:
        pos1, off1 = _shifted(pos0, off0)
    want = torch.full((B, H, W), -7, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_step(p, 2, 2, pos1, off1, z, None, want)
    torch.cuda.synchronize()
    assert int((want >= 0).sum()) == int((steps == 2).sum())
    kernel = torch.cuda._compile_kernel(_LATE_LISTS, "late_lists", compute_capability="100a")
    for cycles in range(0, 20000, 500):
        pos, off = pos0.clone(), off0.clone()
        out = torch.full_like(want, -7)
        torch.cuda.synchronize()
        kernel(grid=(1, 1, 1), block=(64, 1, 1), args=[off1, off, 8, pos1, pos, n, cycles])
        ctx.mulo_redraw_step(p, 2, 2, pos, off, z, None, out)
        assert torch.equal(out, want), cycles


@pytest.mark.parametrize("case", [
    dict(V=8, top_k=3), dict(V=4096, top_k=4095), dict(V=4104, top_k=1), dict(V=8200, top_k=1000), dict(V=16384, top_k=0), dict(V=16392, top_k=2000),
    dict(V=65536, top_k=4000), dict(V=65536, top_k=0), dict(V=32776, top_k=30000, dtype="f32"),
    dict(V=4096, top_k=500, level=-300.0, scale=3.0), dict(V=4096, top_k=500, scale=1e-3), dict(V=8192, top_k=500, quantum=0.5),
    dict(V=16384, top_k=100, scale=0.0), dict(V=20480, top_k=5000, level=5000.0, scale=100.0, dtype="f32"), dict(V=4096, top_k=2100, quantum=0.25),
    dict(V=8192, top_k=700, dtype="f32", cfg_scale=2.0, temperature=0.8),
    # a few entries in a bin whose values lie far apart: past the first histogram's end, above, below, and up to the type's largest
    dict(V=20480, top_k=40, level=3000.0, scale=300.0, dtype="f32"), dict(V=49160, top_k=49100, level=-3000.0, scale=300.0, dtype="f32"),
    dict(V=16384, top_k=20, scale=1e37, dtype="f32"),
], ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_rows_of_all_sizes_and_shapes(ctx, case):
    """Edges of the kernel's pieces and clusters; values outside the first histogram, crowded bins, ties, thresholds below zero."""
    B, H, W, V = 2, 3, 4, case["V"]
    dtype, cfg_scale = case.get("dtype", "bf16"), case.get("cfg_scale", 0.0)
    cfg = synth.RoundConfig("shape", B=B, H=H, W=W, V=V, r=1, dtype=dtype, top_k=case["top_k"], cfg_scale=cfg_scale,
                            temperature=case.get("temperature", 1.0), seed=80)
    g = torch.Generator(device="cuda").manual_seed(V + case["top_k"])
    z = case.get("level", 0.0) + case.get("scale", 2.0) * torch.randn((B, H, W, V), generator=g, device="cuda")
    if "quantum" in case:
        z = (z / case["quantum"]).round() * case["quantum"] + 0.0
        z[..., ::2] = torch.where(z[..., ::2] == 0, -0.0, z[..., ::2])   # both zeros are one value
    cond = z.to(cfg.torch_dtype).contiguous()
    unc = (z + 0.3).to(cfg.torch_dtype).contiguous() if cfg_scale else None
    p = binding.params_from_config(cfg)
    n = B * H * W
    pos, off = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(2 * 3, dtype=torch.int32, device="cuda")
    out = torch.full((B, H, W), -7, dtype=torch.int32, device="cuda")
    ctx.mulo_redraw_plan(p, torch.ones((B, H, W), dtype=torch.int32, device="cuda"), 1, pos, off)
    ctx.mulo_redraw_step(p, 1, 1, pos, off, cond, unc, out)
    for b in range(B):
        want, _, edge = orc.redraw_loop(pu.orc_params(cfg, b), np.ones((H, W), np.int32), [synth.to_numpy_logits(cond[b])],
                                        None if unc is None else [synth.to_numpy_logits(unc[b])], np.zeros((H, W), np.int32), with_edge=True)
        assert not ((out[b].cpu().numpy() != want) & (edge == 0)).any()


@pytest.mark.parametrize("case", [
    dict(V=4096, top_k=500), dict(V=4104, top_k=500), dict(V=8192, top_k=0, dtype="f32"), dict(V=12296, top_k=1500, cfg_scale=3.0, temperature=0.9),
    dict(V=16384, top_k=2000, cfg_scale=3.0), dict(V=16392, top_k=2000), dict(V=24576, top_k=3000, dtype="f32", cfg_scale=1.5),
    dict(V=24584, top_k=0), dict(V=40968, top_k=5000),
], ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_steps_of_more_positions_than_clusters(ctx, case):
    """All 300 positions at once, 33 of them, and one more or less than the clusters of each size: every one is drawn, once, and right."""
    B, H, W, V = 2, 10, 15, case["V"]
    dtype, cfg_scale = case.get("dtype", "bf16"), case.get("cfg_scale", 0.0)
    cfg = synth.RoundConfig("many", B=B, H=H, W=W, V=V, r=1, dtype=dtype, top_k=case["top_k"], cfg_scale=cfg_scale,
                            temperature=case.get("temperature", 1.0), seed=82)
    g = torch.Generator(device="cuda").manual_seed(V)
    z = 2.0 * torch.randn((B, H, W, V), generator=g, device="cuda")
    cond = z.to(cfg.torch_dtype).contiguous()
    unc = (z + 0.3).to(cfg.torch_dtype).contiguous() if cfg_scale else None
    p = binding.params_from_config(cfg)
    n = B * H * W
    pos, off = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(2 * 3, dtype=torch.int32, device="cuda")
    want = None
    for take in (n, 32, 33, 42, 43, 64, 65, 128, 129):
        steps = torch.zeros((B, H, W), dtype=torch.int32, device="cuda")
        steps.view(-1)[:take] = 1
        out = torch.full((B, H, W), -7, dtype=torch.int32, device="cuda")
        ctx.mulo_redraw_plan(p, steps, 1, pos, off)
        ctx.mulo_redraw_step(p, 1, 1, pos, off, cond, unc, out)
        if want is None:
            want = out
            for b in range(B):
                o, _, edge = orc.redraw_loop(pu.orc_params(cfg, b), np.ones((H, W), np.int32), [synth.to_numpy_logits(cond[b])],
                                             None if unc is None else [synth.to_numpy_logits(unc[b])], np.zeros((H, W), np.int32),
                                             with_edge=True)
                assert not ((out[b].cpu().numpy() != o) & (edge == 0)).any()
        got = out.view(-1)
        assert int((got[:take] != want.view(-1)[:take]).sum()) <= 1   # (another order of summation: a draw in 10^4 or fewer)
        assert bool((got[take:] == -7).all())
