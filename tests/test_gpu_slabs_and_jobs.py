"""Attention CTAs that work off several jobs, the layer that leaves for host memory slab by slab, and the ranks of a
small frame's scores, at the sizes where each can go wrong."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import K_FOLD, check_bf16, to_f64, unfold_k
from synthdata import WORKLOADS, make_attention_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_2512_04939_b200 as pkg

    return pkg


def _tokens(n, seed):
    # a common part, as a frame's tokens have: outputs do not average out to their rounding noise
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(1, 1024, generator=g) + 0.5 * torch.randn(n, 1024, generator=g)).to(torch.bfloat16)


def _check_core(name, got, qkv, rows):
    """got[i] is row rows[i] of the attention core over qkv.  The probabilities are rounded to bf16, each off by at most
    2^-9 relative, and the row sum is formed from the rounded values: an output moves by 2^-9 sum_i d_i p_i (v_i - o),
    |d_i| <= 1; Hoeffding's inequality for independent d_i, where 1e7 entries together exceed it with a chance
    of 1e-6 (a factor sqrt(2 ln 2e13) = 7.8)."""
    ref, u, worst = O.attention_core(unfold_k(qkv), heads=16, rows=rows), unfold_k(qkv), 0.0
    for h in range(16):
        q, k, v = (u[:, i * 1024 + h * 64:i * 1024 + h * 64 + 64] for i in range(3))
        s = q[rows] @ k.T / 8.0
        p = np.exp(s - s.max(1, keepdims=True))
        p2 = (p / p.sum(1, keepdims=True)) ** 2
        o = ref[:, h * 64:h * 64 + 64]
        worst = max(worst, float((p2 @ (v * v) - 2 * o * (p2 @ v) + o * o * p2.sum(1, keepdims=True)).max()))
    noise = 7.8 * 2.0 ** -9 * np.sqrt(worst) / float(np.sqrt(np.mean(ref * ref)))
    check_bf16(name, got, ref, noise=noise, sampled=True)


@pytest.mark.parametrize("sharpness", [1.0, 16.0, 64.0])
@pytest.mark.parametrize("frames,grid", [(1, (65, 64)), (2, (64, 64)), (3, (67, 62)), (4, (67, 61))])
def test_sequences_of_several_rounds_of_jobs(lib, frames, grid, sharpness):
    """Frame attention over 4,161 to 4,165 tokens a frame and the global layer over all of them: 17 query blocks, the last with
    one live tile of two, times 16 heads times the frames make 1.8 to 7.4 rounds of 148 CTAs; key tiles with
    and without a second half; all three forms of the softmax, in one CTA after the other."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], 0.0)
    n, t = ctx.n_tokens, ctx.n_tokens // frames
    x = _tokens(n, 11 * frames + grid[1])
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(WORKLOADS["C1"], 6)
    w_qkv[:1024] *= sharpness
    dev = [v.cuda() for v in (w_qkv, b_qkv, w_o, b_o)]
    ctx.global_attn(x.cuda(), *dev)
    ctx.poll()
    qkv, core = to_f64(ctx.debug_buffer(0)), to_f64(ctx.debug_buffer(1))
    rows = np.r_[0:8, n // 2:n // 2 + 8, n - 70:n]
    _check_core(f"global core, {n} rows, sharpness {sharpness}", core[rows], qkv, rows)
    eye = torch.eye(1024, dtype=torch.bfloat16).cuda()  # the output projection hands the core through
    out = to_f64(ctx.frame_attn(x.cuda(), dev[0], dev[1], eye, None))
    ctx.poll()
    rows = np.r_[0:4, t - 70:t]
    for f in range(frames):
        _check_core(f"frame core {f} of {frames}, {t} rows, sharpness {sharpness}", out[f * t + rows], qkv[f * t:(f + 1) * t], rows)
    ctx.close()


@pytest.mark.parametrize("sharpness", [1.0, 16.0, 64.0])
@pytest.mark.parametrize("grid", [(1, 2), (2, 61), (12, 21), (19, 20), (16, 31), (25, 41)])
def test_queries_that_arrive_where_values_will(lib, grid, sharpness):
    """Frames of 7, 127, 257, 385, 501 and 1030 tokens: one to nine key tiles, whose third takes the place of the queries; last
    query tiles of 1 to 127 rows, before the next frame's; all three forms, for which both threads of a row find the same bound."""
    ctx = lib.LiteVGGT(3, grid[0], grid[1], 0.0)
    n, t = ctx.n_tokens, ctx.n_tokens // 3
    x = _tokens(n, 7 * grid[0] + grid[1])
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(WORKLOADS["C1"], 6)
    w_qkv[:1024] *= sharpness
    dev = [v.cuda() for v in (w_qkv, b_qkv, w_o, b_o)]
    ctx.global_attn(x.cuda(), *dev)
    qkv, core = to_f64(ctx.debug_buffer(0)), to_f64(ctx.debug_buffer(1))
    out = to_f64(ctx.frame_attn(x.cuda(), dev[0], dev[1], torch.eye(1024, dtype=torch.bfloat16).cuda(), None))
    ctx.poll()
    rows = np.unique(np.r_[0:min(n, 40), max(0, n - 70):n])
    _check_core(f"global core, {n} rows, sharpness {sharpness}", core[rows], qkv, rows)
    rows = np.unique(np.r_[0:min(t, 20), t // 2, max(0, t - 70):t])
    for f in range(3):
        _check_core(f"frame core {f} of 3, {t} rows, sharpness {sharpness}", out[f * t + rows], qkv[f * t:(f + 1) * t], rows)
    ctx.close()


@pytest.mark.parametrize("entry", ["global", "normed", "frame"])
@pytest.mark.parametrize("value", [2.0 ** 20, 2.0 ** 26, 2.0 ** 100])
def test_large_values_under_a_shifted_reference(lib, entry, value):
    """All keys but the first 64 score what the bound allows, 120, the first ones -45: one reference near the upper limit serves,
    unless the sum over 4,096 or 16,384 keys of 2^(120 - m) times V would not be finite.  All V are equal, so that is what
    every output is."""
    ctx = lib.LiteVGGT(4, 64, 64, 0.0, n_special=0)
    rows = ctx.n_merged
    x, w_qkv, b_qkv = (torch.zeros(*s, dtype=torch.bfloat16) for s in ((rows, 1024), (3072, 1024), (3072,)))
    u = torch.tensor([1.0, -1.0] * 32)
    first = u.clone()
    first[:44] *= -1.0  # 12 of 32 pairs more that point the other way than along
    x[:, :64], x[:, 64] = u, value
    x.view(4, -1, 1024)[:, :64, :64] = first
    scale = 10.375  # times 64 / 8 log2 e = 119.7
    for h in range(16):
        w_qkv[1024 + 64 * h + torch.arange(64), torch.arange(64)] = 1.0
        w_qkv[2048 + 64 * h, 64] = 1.0
        b_qkv[64 * h:64 * h + 64] = u if entry == "normed" else scale * u
    eye, one, zero = torch.eye(1024, dtype=torch.bfloat16), torch.ones(64, dtype=torch.bfloat16), torch.zeros(64, dtype=torch.bfloat16)
    dev = [t.cuda() for t in (x, w_qkv, b_qkv, eye)]
    if entry == "frame":
        out = ctx.frame_attn(*dev, None)
    elif entry == "global":
        out = ctx.global_attn(*dev, None)
    else:
        out = ctx.global_attn_ext(None, *dev, None, q_norm=((scale * one).cuda(), zero.cuda()), k_norm=(one.cuda(), zero.cuda()))
    ctx.poll()
    assert (out[:, ::64].float() == value).all()
    ctx.close()


@pytest.mark.parametrize("frames,many,top,bound", [(2, 3900, 63.0, 243.0), (17, 30000, 66.0, 239.0)])
def test_parts_of_a_row_under_references_far_apart(lib, frames, many, top, bound):
    """8,192 rows, where some jobs are split in two along the keys, and 69,632 in two key chunks.  The first half scores -18 in
    its first 64 keys, so that the running maximum has to serve, and 51 in `many` later ones, which is not beyond what a
    reference near the first maximum takes; the second half's first key scores `top` and one reference over 130 binades higher
    serves it.  The first half holds about half of every row, the only part with
    V = 1.  Scores are equal within a half, so an output is off by the rounding of two probabilities and its own: 3 x 2^-9 of it."""
    ctx = lib.LiteVGGT(frames, 64, 64, 0.0, n_special=0)
    rows = ctx.n_merged
    half = rows // 2
    x, w_qkv, b_qkv, w_o, b_o = (torch.zeros(*s, dtype=torch.bfloat16) for s in ((rows, 1024), (3072, 1024), (3072,), (1024, 1024), (1024,)))
    score = torch.full((rows,), -50.0)
    score[0], score[64:64 + many], score[half] = -18.0, 51.0, top
    x[:, 0] = score / 16 / K_FOLD
    x[5, 1] = (bound ** 2 - 50.0 ** 2) ** 0.5 / 16 / K_FOLD  # a long key, across the queries but for its score of -50
    x[64:64 + many, 2] = 1.0
    for h in range(16):
        b_qkv[64 * h] = 16.0
        w_qkv[1024 + 64 * h, 0] = w_qkv[1024 + 64 * h + 1, 1] = w_qkv[2048 + 64 * h, 2] = 1.0
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    s = 16.0 * to_f64(ctx.debug_buffer(0)[:, 1024:1025])[:, 0]  # the scores that the kernel had, in base 2
    p = np.exp2(s - s.max())
    ref = p[64:64 + many].sum() / p.sum()
    out = to_f64(ctx.debug_buffer(1)[:, ::64])
    assert 0.2 < ref < 0.6 and np.abs(out / ref - 1.0).max() <= 3 * 2.0 ** -9
    ctx.close()


def _check_up_to_rounding(name, got, ref, x):
    got, ref = got.float(), ref.float()
    gap = (got - ref).abs()
    # a bf16 unit of either value, and of the attention output before the residual was added
    unit = 2.0 ** -7 * torch.maximum(ref.abs(), (ref - x.float()).abs())
    assert bool((gap <= 2 * unit + 1e-3).all()), f"{name}: {gap.max()}"
    assert float((gap != 0).float().mean()) < 0.2


@pytest.mark.parametrize("frames,grid,ratio", [
    (3, (37, 37), 0.0),    # 4,122 rows: the fewest that leave in slabs, two of them
    (5, (37, 37), 0.3),    # a second slab of two rounds, not full
    (9, (37, 37), 0.45),   # anchors of the first frame that stand for many tokens
    (16, (37, 28), 0.42)])  # several whole slabs
def test_output_that_leaves_in_slabs(lib, frames, grid, ratio):
    """Calls in a row, the plan rebuilt in place right behind each: every output is the ordered entry's for the plan
    the call was given (jobs of the last round are split elsewhere: one rounding of y and one of the output apart),
    also into pageable memory and at an address that 16-byte stores do not fit."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], ratio)
    n = ctx.n_tokens
    w = [v.cuda() for v in make_attention_weights(WORKLOADS["C1"], 2)]
    g = torch.Generator().manual_seed(n)
    grads = [torch.rand(frames, *grid, generator=g).cuda() for _ in range(3)]
    xs = [_tokens(n, n + i).pin_memory() for i in range(3)]
    expected = []
    plan = None
    for x, grad in zip(xs, grads):
        out = torch.empty_like(x).pin_memory()
        plan = ctx.global_layer_host(plan, x, *w, out, grad=grad)
        ctx.poll()
        expected.append(out)
    odd = torch.zeros(n * 1024 + 1, dtype=torch.bfloat16).pin_memory()[1:].view(n, 1024)
    outs = [torch.zeros_like(xs[0]).pin_memory(), odd, torch.zeros_like(xs[0])]
    for order in ((0, 1, 2), (2, 0, 1)):
        for x, grad, k in zip(xs, grads, order):
            outs[k].zero_()
            ctx.global_layer_host_pipelined(plan, x, *w, outs[k], grad=grad)
            if outs[k].is_pinned():
                ctx.merge_plan(_tokens(n, 7).cuda(), grads[0], plan)  # what is still on its way keeps the plan it had
        ctx.host_drain()
        ctx.poll()
        for i, k in enumerate(order):
            _check_up_to_rounding(f"call {i}", outs[k], expected[i], xs[i])
    plan.destroy()
    ctx.close()


def test_host_entries_in_turn_without_a_drain(lib):
    """An ordered call right behind a pipelined one, and the other way round, more often than there are buffers: every output is
    what the call gives alone.  The first pipelined call leaves in slabs, those behind it as the ordered ones do."""
    frames, grid = 5, (37, 37)
    ctx = lib.LiteVGGT(frames, *grid, 0.3)
    n = ctx.n_tokens
    w = [v.cuda() for v in make_attention_weights(WORKLOADS["C1"], 2)]
    g = torch.Generator().manual_seed(n)
    xs = [_tokens(n, n + i).pin_memory() for i in range(6)]
    plan = ctx.merge_plan(xs[0].cuda(), torch.rand(frames, *grid, generator=g).cuda())
    calls = (ctx.global_layer_host_pipelined, ctx.global_layer_host)
    alone = []
    for call in calls:
        outs = [torch.zeros_like(x).pin_memory() for x in xs]
        for x, out in zip(xs, outs):
            before = ctx.launch_count()
            call(plan, x, *w, out)
            launches = ctx.launch_count() - before
            ctx.host_drain()
            ctx.poll()
        alone.append((launches, outs))
    assert alone[0][0] > alone[1][0] and not torch.equal(alone[0][1][0], alone[1][1][0])  # slabs, and a whole
    for i, (a, b) in enumerate(zip(alone[0][1], alone[1][1])):  # out of either of the two buffers
        _check_up_to_rounding(f"call {i} and its drain", a, b, xs[i])
    for order in ((0, 1, 0, 1, 1, 0), (1, 0, 0, 1, 0, 0)):
        outs = [torch.zeros_like(x).pin_memory() for x in xs]
        for k, x, out in zip(order, xs, outs):
            calls[k](plan, x, *w, out)
        ctx.host_drain()
        ctx.poll()
        first = order.index(0)
        for i, out in enumerate(outs):
            assert torch.equal(out, alone[0 if i == first else 1][1][i]), f"call {i} of {order}"
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("grid,keep", [((1, 1), 0.1), ((16, 16), 0.1), ((16, 16), 0.9), ((4, 64), 0.5), ((7, 37), 0.1), ((6, 43), 0.3)])
def test_ranks_of_a_small_frames_scores(lib, grid, keep):
    """Frames of 1, 256, 258 and 259 patches: up to 256 every patch is ranked against the others, above a search finds
    the threshold.  Scores in few steps, so that ties decide."""
    ctx = lib.LiteVGGT(4, grid[0], grid[1], 0.3, ga_keep_frac=keep)
    g = torch.Generator().manual_seed(grid[0] * 100 + grid[1])
    x = torch.randn(13, 1024, generator=g)[torch.randint(0, 13, (ctx.n_tokens,), generator=g)].to(torch.bfloat16)
    grad = torch.randint(0, 4, (4, *grid), generator=g).float()
    plan = ctx.merge_plan(x.cuda(), grad.cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    assert np.array_equal(ex["cls"], O.partition(ex["ga"], ga_keep_frac=keep))
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("above", [88.5, 95.0, 97.5])
def test_reference_that_serves_a_whole_sweep_at_its_limits(lib, above):
    """16,384 rows: one reference serves score bounds up to 92 over it, and a known score up to 88 under it.  Keys 0 and 1
    score 0, the highest; key 1 is long, across the queries, so that the bound lies 84 + `above` over it: under 96 the reference
    serves, above the running maximum has to.  The other keys sit 40 binades down with V = 1 where keys 0 and 1
    have V = 0: the output is what they hold together, 2^-27, and an error of 2^-24 of the row's mass is allowed."""
    rows = 16384
    ctx = lib.LiteVGGT(4, 64, 64, 0.0, n_special=0)
    assert ctx.n_merged == rows
    x, w_qkv, b_qkv, w_o, b_o = (torch.zeros(*s, dtype=torch.bfloat16) for s in ((rows, 1024), (3072, 1024), (3072,), (1024, 1024), (1024,)))
    x[2:, 0], x[1, 1], x[2:, 2] = -40.0 / 16 / K_FOLD, (84 + above) / 16 / K_FOLD, 1.0
    for h in range(16):
        b_qkv[64 * h] = 16.0
        w_qkv[1024 + 64 * h, 0] = w_qkv[1024 + 64 * h + 1, 1] = w_qkv[2048 + 64 * h, 2] = 1.0
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    out = to_f64(ctx.debug_buffer(1))[:, ::64]
    assert np.isfinite(out).all() and np.abs(out - (rows - 2) * 2.0 ** -41).max() <= 2.0 ** -24
    ctx.close()


@pytest.mark.parametrize("bound", [170.0, 179.0, 185.0])
def test_reference_far_below_the_scores_does_not_overflow(lib, bound):
    """16,384 rows whose first 64 keys score 0 and all others `bound`, the largest that the lengths allow: the reference
    lies 92 under them (or is a running one, above 180), their probabilities of 2^92 and values of 2^20 add up to 2^126
    before the division, and the output is 2^20."""
    rows = 16384
    ctx = lib.LiteVGGT(4, 64, 64, 0.0, n_special=0)
    x, w_qkv, b_qkv, w_o, b_o = (torch.zeros(*s, dtype=torch.bfloat16) for s in ((rows, 1024), (3072, 1024), (3072,), (1024, 1024), (1024,)))
    x[64:, 0], x[64:, 2] = bound / 16 / K_FOLD, 2.0 ** 20
    for h in range(16):
        b_qkv[64 * h] = 16.0
        w_qkv[1024 + 64 * h, 0] = w_qkv[2048 + 64 * h, 2] = 1.0
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    out = to_f64(ctx.debug_buffer(1))[:, ::64]
    assert np.isfinite(out).all() and np.abs(out / 2.0 ** 20 - 1).max() <= 2.0 ** -8
    ctx.close()
