"""GPU parity: every step of the CUDA path against the CPU oracle on the same seeded
inputs, through the C ABI.  Integer / index work must be bit-exact given the same
upstream result; floating point obeys the tolerances written beside each check."""
import numpy as np
import pytest
import torch

import oracle as O
from synthdata import (WORKLOADS, Workload, make_attention_weights, make_block_weights, make_images,
                       make_peaked_attention_inputs, make_tokens)
from helpers import (CORE_NOISE, K_FOLD, LAYER_NOISE, bf16_bound, bf16_round, check_bf16, fold_k, rel_err, report,
                     to_f64, unfold_k)

pytestmark = pytest.mark.gpu

MID = Workload("MID", 8, 16, 16, 0.3, "polygons", 1, 6, 7000)      # N=2088, M=1462: 12 key tiles, ragged
ODD = Workload("ODD", 5, 9, 11, 0.45, "polygons", 1, 6, 8000)       # odd grid: clipped cells, tiny tail


@pytest.fixture(scope="module")
def lib():
    import paper_2512_04939_b200 as pkg
    return pkg


def _ctx(lib, wl, **kw):
    return lib.LiteVGGT(wl.frames, wl.grid_h, wl.grid_w, wl.merge_ratio, **kw)


_CACHE = {}


def _inputs(wl):
    if wl.name not in _CACHE:
        img = make_images(wl)
        tok = make_tokens(wl, img)
        _CACHE[wl.name] = (img, tok)
    return _CACHE[wl.name]


_PLANS = {}


def _oracle_plan(wl):
    if wl.name not in _PLANS:
        img, tok = _inputs(wl)
        grad = O.grad_map(img.numpy())
        _PLANS[wl.name] = (grad, O.merge_plan(to_f64(tok), grad, wl.frames, wl.grid_h, wl.grid_w,
                                               merge_ratio=wl.merge_ratio))
    return _PLANS[wl.name]


# ------------------------------------------------------------------ a1 grad map
@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD, WORKLOADS["C2"]], ids=lambda w: w.name)
def test_grad_map(lib, wl):
    img, _ = _inputs(wl)
    ctx = _ctx(lib, wl)
    got = ctx.grad_map(img.cuda())
    ctx.poll()
    ref = O.grad_map(img.numpy())
    # fp32 arithmetic on O(1) values, 196-term means: 1e-5 relative to the map's scale
    assert np.abs(to_f64(got) - ref).max() <= 1e-5 * max(ref.max(), 1e-3)
    ctx.close()


# ------------------------------------------------------------------ a2/a3 scoring + partition
@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD, MID], ids=lambda w: w.name)
def test_var_map_and_partition(lib, wl):
    img, tok = _inputs(wl)
    grad, ref = _oracle_plan(wl)
    ctx = _ctx(lib, wl)
    plan = ctx.merge_plan(tok.cuda(), torch.from_numpy(grad.astype(np.float32)).cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    # Var map: fp32 two-pass variance vs float64, relative to the map's scale
    assert np.abs(ex["var"] - ref["var"]).max() <= 2e-5 * ref["var"].max()
    assert np.abs(ex["ga"] - ref["ga"]).max() <= 1e-5
    # classes: the per-frame counts are exact; tokens may differ only where the deciding
    # score gap is below 1e-5 (fp32 vs fp64 scores), and 99.9 % must agree overall
    cls = ex["cls"]
    sz = ref["sizes"]
    per_frame = cls.reshape(wl.frames, -1)
    assert np.all(per_frame[:, :5] == O.CLS_PROTECTED)
    assert np.all(per_frame[0, 5:] == O.CLS_DST)
    for f in range(1, wl.frames):
        assert (per_frame[f] == O.CLS_DST).sum() == sz["n_dst_frame"]
        assert (per_frame[f] == O.CLS_GA).sum() == sz["n_ga_frame"]
        assert (per_frame[f] == O.CLS_SRC).sum() == sz["n_src_frame"]
    diff = np.flatnonzero(cls != ref["cls"])
    assert diff.size <= 1e-3 * cls.size
    if diff.size:
        ga = ref["ga"].reshape(wl.frames, -1)
        for i in diff:
            f, t = divmod(int(i), wl.tokens_per_frame)
            others = np.delete(ga[f], t - 5)
            assert np.abs(others - ga[f, t - 5]).min() < 1e-5, "class differs without a near-tie"
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("patch,grid_h,grid_w", [(8, 9, 7), (16, 5, 6), (30, 3, 4), (1, 6, 33)])
def test_grad_map_other_patch_sizes(lib, patch, grid_h, grid_w):
    """Patch sizes other than 14: three patches per strip, one per strip, the largest accepted size and
    single-pixel patches (the Grad map is then the Sobel magnitude itself)."""
    g = torch.Generator().manual_seed(100 + patch)
    img = torch.rand(3, 3, grid_h * patch, grid_w * patch, generator=g)
    ctx = lib.LiteVGGT(3, grid_h, grid_w, 0.5, patch_px=patch)
    got = ctx.grad_map(img.cuda())
    ctx.poll()
    ref = O.grad_map(img.numpy(), patch_px=patch)
    assert got.shape == ref.shape
    assert np.abs(to_f64(got) - ref).max() <= 1e-5 * max(ref.max(), 1e-3)
    ctx.close()


def test_scoring_maps_on_the_widest_grid(lib):
    """Grid of 33 x 64 patches: the widest row the library accepts (the Var map's per-row results and
    the Grad map's strips reach their limits), more than one block of 30 grid rows, and a frame whose
    last strip holds two patches exactly."""
    wl = Workload("WIDE", 2, 33, 64, 0.5, "polygons", 1, 6, 9000)
    img = make_images(wl)
    tok = make_tokens(wl, img)
    ctx = _ctx(lib, wl)
    grad = ctx.grad_map(img.cuda())
    ref_grad = O.grad_map(img.numpy())
    assert np.abs(to_f64(grad) - ref_grad).max() <= 1e-5 * max(ref_grad.max(), 1e-3)
    plan = ctx.merge_plan(tok.cuda(), grad)
    ctx.poll()
    ex = ctx.plan_export(plan)
    ref_var = O.var_map(to_f64(tok), wl.frames, wl.grid_h, wl.grid_w)
    assert np.abs(ex["var"] - ref_var).max() <= 2e-5 * ref_var.max()
    plan.destroy()
    ctx.close()


# ------------------------------------------------------------------ a4 matching (stage-isolated)
def _check_match(ex, ref):
    agree = ex["best_dst"] == ref["best_dst"]
    margin = ref["best_sim"] - ref["second_sim"]
    assert np.all(agree[margin > 1e-3]), "argmax differs although the oracle's margin exceeds 1e-3"
    assert agree.mean() >= 0.999
    # a differing index must still be a near-tie: its similarity within 1e-5 of the best
    assert np.abs(ex["best_sim"] - ref["best_sim"]).max() <= 1e-5
    return agree.mean(), margin


@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD, MID], ids=lambda w: w.name)
def test_match_with_oracle_partition(lib, wl):
    _, tok = _inputs(wl)
    _, ref = _oracle_plan(wl)
    ctx = _ctx(lib, wl)
    plan = ctx.merge_plan_with_partition(tok.cuda(), torch.from_numpy(ref["cls"]).cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    _check_match(ex, ref)
    plan.destroy()
    ctx.close()


# ------------------------------------------------------------------ a5 selection + index arrays
@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD, MID], ids=lambda w: w.name)
def test_index_build_bit_exact_given_same_matches(lib, wl):
    _, tok = _inputs(wl)
    _, ref = _oracle_plan(wl)
    ctx = _ctx(lib, wl)
    plan = ctx.merge_plan_with_partition(tok.cuda(), torch.from_numpy(ref["cls"]).cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    dst_of, size, kept = O.select_and_index(ref["cls"], ex["best_dst"], ex["best_sim"], ref["sizes"]["R"])
    assert np.array_equal(ex["dst_of"], dst_of)
    assert np.array_equal(ex["size"], size)
    assert np.array_equal(ex["kept_idx"], kept)
    # and when the matches agree with the oracle's, so does the whole plan
    if np.array_equal(ex["best_dst"], ref["best_dst"]) and ref["sizes"]["R"] == ref["sizes"]["n_src"]:
        assert np.array_equal(ex["dst_of"], ref["dst_of"])
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("frames,grid,ratio,cell,kind", [
    (38, (16, 16), 0.3, 2, "random"),
    (7, (19, 25), 0.45, 2, "tied"),     # ties at the threshold, one block
    (35, (16, 16), 0.45, 2, "tied"),    # ties across the cluster's blocks
    (16, (15, 21), 0.45, 2, "tied"),    # 5,120 tokens: the most for one block, two chunks of tokens
    (16, (15, 21), 1.0, 16, "random"),  # and the most shared memory
    (3, (46, 37), 0.45, 2, "tied"),     # 5,121: the smallest cluster
    (31, (28, 37), 0.3, 2, "random"),   # 32,271 tokens: the largest
    (31, (28, 37), 0.0, 2, "random"),   # nothing merged
    (14, (37, 37), 0.5, 16, "equal"),   # one segment of 9,618 tokens
    (24, (37, 37), 0.3, 2, "tied"),     # 32,976 tokens: the smallest as launches
    (24, (37, 37), 1.0, 2, "random"),   # every src token merged
    (24, (37, 37), 0.0, 2, "random"),
    (30, (37, 37), 0.5, 16, "equal"),   # one segment of 20,610 tokens
    (71, (37, 37), 0.3, 2, "tied"),     # 97,554 tokens: the most that the cluster numbers
    (72, (37, 37), 0.3, 2, "tied"),     # 98,928: the fewest that launches do, ties across chunks
    (72, (37, 37), 1.0, 2, "random"),   # every src token merged
    (72, (37, 37), 0.5, 16, "equal"),   # one segment of 49,464 tokens, walked by one block
    (72, (37, 37), 0.0, 2, "random"),   # nothing merged
    (12, (20, 20), 0.5, 1, "random"),   # every patch an anchor, so no src token: one block,
    (31, (28, 37), 0.5, 1, "random"),   # one cluster,
    (24, (37, 37), 0.5, 1, "random"),   # the cluster and launches,
    (72, (37, 37), 0.5, 1, "random")])  # launches
def test_index_arrays_at_the_limits_of_their_forms(lib, frames, grid, ratio, cell, kind):
    """Numbers and sizes against the oracle's on the library's own matches; segments by a merge, whose sums show their order."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], ratio, cell_h=cell, cell_w=cell)
    n = ctx.n_tokens
    g = torch.Generator().manual_seed(n + frames)
    if kind == "random":
        x = torch.randn(n, 1024, generator=g)
    elif kind == "tied":
        x = torch.randn(13, 1024, generator=g)[torch.randint(0, 13, (n,), generator=g)]
    else:  # one direction, so that the first anchor takes all
        x = torch.ones(n, 1024) * 2.0 ** torch.randint(-3, 4, (n, 1), generator=g)
    x = x.to(torch.bfloat16).cuda()
    plan = ctx.merge_plan(x, torch.rand(frames, *grid, generator=g).cuda())
    ctx.merge_plan(x, torch.rand(frames, *grid, generator=g).cuda(), plan)
    ctx.poll()
    ex = ctx.plan_export(plan)
    dst_of, size, kept = O.select_and_index(ex["cls"], ex["best_dst"], ex["best_sim"], n - ctx.n_merged)
    assert np.array_equal(ex["dst_of"], dst_of) and np.array_equal(ex["size"], size) and np.array_equal(ex["kept_idx"], kept)
    rows = x[:, :32].float().cpu().numpy()
    total, rest = rows[kept], np.setdiff1d(np.arange(n), kept)
    np.add.at(total, dst_of[rest], rows[rest])  # one after the other, in ascending order
    want = torch.from_numpy(total / size[:, None].astype(np.float32)).to(torch.bfloat16)
    assert torch.equal(ctx.merge(plan, x)[:, :32].cpu(), want)
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("frames,grid,ratio,cell,keep,kind", [
    (1, (5, 7), 0.5, 2, 0.1, "random"),     # no src token
    (2, (9, 9), 0.3, 2, 0.6, "random"),     # few src tokens, all of them merged
    (5, (9, 11), 0.45, 2, 0.1, "tied"),     # every cosine equal to many others
    (7, (19, 25), 0.45, 2, 0.0, "equal"),   # one anchor takes 1512 tokens: a long segment, single block
    (6, (35, 39), 0.2, 8, 0.1, "tied"),     # 8,220 tokens: one cluster
    (9, (37, 37), 0.45, 2, 0.1, "random"),  # one cluster; 28 row blocks, fewer than pairs: all in column runs
    (30, (37, 37), 0.5, 2, 0.1, "random"),  # cluster and launches; 25,288 src tokens: a whole sweep of the 74 pairs, 25 row blocks in column runs
    (8, (37, 37), 1.0, 16, 0.0, "equal")])  # one cluster, one segment of 9,583, every src token merged
def test_partition_and_index_build_on_degenerate_inputs(lib, frames, grid, ratio, cell, keep, kind):
    """Ties everywhere, segments longer than a block ranks by comparison, everything or nothing merged."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], ratio, cell_h=cell, cell_w=cell, ga_keep_frac=keep)
    n = ctx.n_tokens
    g = torch.Generator().manual_seed(n)
    if kind == "random":
        x, grad = torch.randn(n, 1024, generator=g), torch.rand(frames, *grid, generator=g)
    elif kind == "tied":
        x = torch.randn(13, 1024, generator=g)[torch.randint(0, 13, (n,), generator=g)]
        grad = torch.randint(0, 3, (frames, *grid), generator=g).float()
    else:
        x, grad = torch.ones(n, 1024), torch.zeros(frames, *grid)
    x = x.to(torch.bfloat16)
    plan = ctx.merge_plan(x.cuda(), grad.cuda())
    ctx.merge_plan(x.cuda(), grad.cuda(), plan)  # and once more in place
    ctx.poll()
    ex = ctx.plan_export(plan)
    assert np.array_equal(ex["cls"], O.partition(ex["ga"], ga_keep_frac=keep, cell_h=cell, cell_w=cell))
    removed = n - ctx.n_merged
    dst_of, size, kept = O.select_and_index(ex["cls"], ex["best_dst"], ex["best_sim"], removed)
    assert np.array_equal(ex["dst_of"], dst_of)
    assert np.array_equal(ex["size"], size)
    assert np.array_equal(ex["kept_idx"], kept)
    src, dst = np.flatnonzero(ex["cls"] == O.CLS_SRC), np.flatnonzero(ex["cls"] == O.CLS_DST)
    if src.size:
        rows = np.arange(src.size) if src.size < 2048 else np.r_[0:512, src.size - 512:src.size]
        if src.size > 19072:  # and where the whole sweeps end: row 74 * 256
            rows = np.r_[0:256, 18816:19072, src.size - 512:src.size]
        best, sim, second = O.match(to_f64(x), src, dst, rows=rows)
        if kind != "random":  # equal rows have equal products: the lowest anchor wins every tie
            assert np.array_equal(to_f64(x)[ex["best_dst"][rows]], to_f64(x)[best])
            assert (ex["best_dst"][rows] <= best).all()
        else:
            assert np.array_equal(ex["best_dst"][rows][sim - second > 1e-5], best[sim - second > 1e-5])
    # the segments hold their tokens in ascending order: the mean of a row is summed in that order
    xm = ctx.merge(plan, x.cuda())
    ctx.poll()
    if kind == "equal":
        assert bool((xm == 1).all())
    plan.destroy()
    ctx.close()


def test_identity_at_ratio_zero_and_reuse_equals_recompute(lib):
    wl = WORKLOADS["C1"]
    img, tok = _inputs(wl)
    grad = torch.from_numpy(O.grad_map(img.numpy()).astype(np.float32)).cuda()
    x = tok.cuda()
    ctx0 = lib.LiteVGGT(wl.frames, wl.grid_h, wl.grid_w, 0.0)
    p0 = ctx0.merge_plan(x, grad)
    ex = ctx0.plan_export(p0)
    assert ctx0.n_merged == ctx0.n_tokens and np.array_equal(ex["dst_of"], np.arange(ctx0.n_tokens))
    assert torch.equal(ctx0.merge(p0, x), x)
    ctx0.poll()
    p0.destroy(); ctx0.close()
    ctx = _ctx(lib, wl)
    p = ctx.merge_plan(x, grad)
    a = ctx.plan_export(p)
    ctx.merge_plan(x, grad, p)  # refresh in place on unchanged features
    b = ctx.plan_export(p)
    for k in ("dst_of", "size", "kept_idx", "cls", "best_dst"):
        assert np.array_equal(a[k], b[k]), k
    assert [l for l in range(24) if ctx.should_refresh(p, l)] == [0, 6, 12, 18]
    assert ctx.should_refresh(None, 3)
    ctx.poll()
    p.destroy(); ctx.close()


# ------------------------------------------------------------------ naive (fixed-stride) anchors
def test_fixed_stride_anchor_rule(lib):
    """The partition the paper argues against (Sec. 3.2: fixed-stride dst tokens, nothing protected)
    is the same code path with the GA map switched off: alpha = beta = 0 makes every score tie, ties
    go to the lowest index, so each 2x2 cell's anchor is its top-left token; ga_keep_frac = 0 leaves
    no GA tokens."""
    wl = ODD
    img, tok = _inputs(wl)
    grad = O.grad_map(img.numpy())
    ref = O.merge_plan(to_f64(tok), grad, wl.frames, wl.grid_h, wl.grid_w, merge_ratio=wl.merge_ratio,
                       ga_keep_frac=0.0, alpha=0.0, beta=0.0)
    ctx = lib.LiteVGGT(wl.frames, wl.grid_h, wl.grid_w, wl.merge_ratio, ga_keep_frac=0.0, alpha=0.0, beta=0.0)
    assert (ctx.n_src, ctx.n_dst, ctx.n_merged) == (ref["sizes"]["n_src"], ref["sizes"]["n_dst"], ref["sizes"]["M"])
    plan = ctx.merge_plan(tok.cuda(), torch.from_numpy(grad.astype(np.float32)).cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    assert np.array_equal(ex["cls"], ref["cls"])
    per_frame = ex["cls"].reshape(wl.frames, wl.tokens_per_frame)[1:, 5:].reshape(-1, wl.grid_h, wl.grid_w)
    assert not np.any(per_frame == O.CLS_GA)
    assert np.all(per_frame[:, ::2, ::2] == O.CLS_DST) and (per_frame == O.CLS_DST).sum() == (wl.frames - 1) * 5 * 6
    _check_match(ex, ref)
    dst_of, size, kept = O.select_and_index(ref["cls"], ex["best_dst"], ex["best_sim"], ref["sizes"]["R"])
    assert np.array_equal(ex["dst_of"], dst_of) and np.array_equal(ex["size"], size)
    plan.destroy()
    ctx.close()


def test_seeded_random_anchor_rule(lib):
    """The other naive partition (Sec. 3.2): one anchor per 2x2 cell drawn at random from a seeded
    generator, nothing protected.  The classes are made on the host (the oracle's partition fed with
    random scores) and handed to the library, which matches, selects and merges with them; everything
    downstream is checked against the oracle on the same classes."""
    wl = ODD
    _, tok = _inputs(wl)
    scores = np.random.default_rng(424242).random((wl.frames, wl.grid_h, wl.grid_w))
    cls = O.partition(scores, ga_keep_frac=0.0)
    fixed = O.partition(np.zeros_like(scores), ga_keep_frac=0.0)
    assert (cls != fixed).any() and not np.any(cls == O.CLS_GA)
    x64 = to_f64(tok)
    src_idx, dst_idx = np.flatnonzero(cls == O.CLS_SRC), np.flatnonzero(cls == O.CLS_DST)
    best_dst, sim1, sim2 = O.match(x64, src_idx, dst_idx)
    ctx = lib.LiteVGGT(wl.frames, wl.grid_h, wl.grid_w, wl.merge_ratio, ga_keep_frac=0.0)
    assert (ctx.n_src, ctx.n_dst) == (src_idx.size, dst_idx.size)
    x = tok.cuda()
    plan = ctx.merge_plan_with_partition(x, torch.from_numpy(cls).cuda())
    ctx.poll()
    ex = ctx.plan_export(plan)
    assert np.array_equal(ex["cls"], cls)
    _check_match(ex, dict(best_dst=best_dst, best_sim=sim1, second_sim=sim2))
    n_remove = O.derived_sizes(wl.frames, wl.grid_h, wl.grid_w, merge_ratio=wl.merge_ratio, ga_keep_frac=0.0)["R"]
    dst_of, size, kept = O.select_and_index(cls, ex["best_dst"], ex["best_sim"], n_remove)
    assert np.array_equal(ex["dst_of"], dst_of) and np.array_equal(ex["size"], size)
    assert np.array_equal(ex["kept_idx"], kept)
    xm = ctx.merge(plan, x)
    ctx.poll()
    ref_m = O.merge(x64, dst_of, ctx.n_merged)
    assert rel_err(to_f64(xm), ref_m) <= bf16_bound(ref_m)
    plan.destroy()
    ctx.close()


# ------------------------------------------------------------------ a6 / a10 merge, unmerge
@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD, MID], ids=lambda w: w.name)
def test_merge_unmerge_with_oracle_plan(lib, wl):
    _, tok = _inputs(wl)
    _, ref = _oracle_plan(wl)
    ctx = _ctx(lib, wl)
    plan = ctx.plan_import(ref["dst_of"])
    x = tok.cuda()
    xm = ctx.merge(plan, x)
    ctx.poll()
    x64 = to_f64(tok)
    ref_m = O.merge(x64, ref["dst_of"], ref["sizes"]["M"])
    got = to_f64(xm)
    check_bf16(f"{wl.name}: merge", got, ref_m)
    single = ref["size"] == 1
    assert np.array_equal(got[single], x64[ref["kept_idx"][single]])  # bit-exact copies
    # conservation of size-weighted sums, up to the one bf16 rounding per merged row
    lhs = (ref["size"][:, None] * got).sum(0)
    assert np.abs(lhs - x64.sum(0)).max() <= 2.0 ** -8 * np.abs(x64).sum(0).max()
    # unmerge: pure gather is bit-exact; with residual one fp32 add + rounding
    ym = torch.randn(ctx.n_merged, 1024, generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    out = ctx.unmerge(plan, ym)
    assert np.array_equal(to_f64(out), O.unmerge(to_f64(ym), ref["dst_of"]))
    out_r = ctx.unmerge(plan, ym, x)
    ref_r = O.unmerge(to_f64(ym), ref["dst_of"], x64)
    check_bf16(f"{wl.name}: unmerge with residual", to_f64(out_r), ref_r)
    ctx.poll()
    plan.destroy()
    ctx.close()


# ------------------------------------------------------------------ a7 / a9 projections
@pytest.mark.parametrize("m,k,n", [(543, 1024, 3072), (1462, 1024, 1024), (5, 64, 64), (300, 128, 320)])
def test_linear(lib, m, k, n):
    wl = WORKLOADS["C1"]
    ctx = _ctx(lib, wl)
    g = torch.Generator().manual_seed(m + n)
    a = torch.randn(m, k, generator=g).to(torch.bfloat16)
    w = (0.05 * torch.randn(n, k, generator=g)).to(torch.bfloat16)
    b = (0.1 * torch.randn(n, generator=g)).to(torch.bfloat16)
    for bias in (b, None):
        got = ctx.linear(a.cuda(), w.cuda(), None if bias is None else bias.cuda())
        ctx.poll()
        ref = to_f64(a) @ to_f64(w).T + (0 if bias is None else to_f64(bias))
        check_bf16(f"linear {m}x{k}x{n}", to_f64(got), ref)
    ctx.close()


@pytest.mark.parametrize("m,k,n", [(1848, 1024, 1344), (2305, 512, 2112), (3360, 1024, 2048), (3700, 1024, 4096), (3700, 4096, 832),
                                   (2305, 768, 2112)])
def test_linear_on_tiles_that_end_within_64_columns(lib, m, k, n):
    """Tiles of 160 and 224 columns: 64, 32, 64, 160 and 32 are left for the last one, whole chunks of 64 and halves (and 192 columns
    at k = 512)."""
    ctx = _ctx(lib, WORKLOADS["C1"])
    g = torch.Generator().manual_seed(m + n)
    a = torch.randn(m, k, generator=g).to(torch.bfloat16)
    w = (0.05 * torch.randn(n, k, generator=g)).to(torch.bfloat16)
    b = (0.1 * torch.randn(n, generator=g)).to(torch.bfloat16)
    rows = np.unique(np.r_[0:40, 100:160, 250:260, m - 70:m])
    for bias in (b, None):
        got = ctx.linear(a.cuda(), w.cuda(), None if bias is None else bias.cuda())
        ctx.poll()
        ref = to_f64(a)[rows] @ to_f64(w).T + (0 if bias is None else to_f64(bias))
        check_bf16(f"linear {m}x{k}x{n}", to_f64(got)[rows], ref, sampled=True)
    ctx.close()


def test_mlp_in_place_on_tiles_that_end_within_64_columns(lib):
    """3,360 rows, whose second layer has tiles of 224 columns; the residual where the output goes."""
    ctx = lib.LiteVGGT(7, 19, 25, 0.45)
    g = torch.Generator().manual_seed(5)
    x = torch.randn(3360, 1024, generator=g).to(torch.bfloat16)
    w1, w2 = (0.02 * torch.randn(4096, 1024, generator=g)).to(torch.bfloat16), (0.02 * torch.randn(1024, 4096, generator=g)).to(torch.bfloat16)
    b1, b2 = (0.1 * torch.randn(4096, generator=g)).to(torch.bfloat16), (0.1 * torch.randn(1024, generator=g)).to(torch.bfloat16)
    y = x.cuda()
    ctx.mlp(y, w1.cuda(), b1.cuda(), w2.cuda(), b2.cuda(), residual=y, out=y)
    ctx.poll()
    rows = np.r_[0:20, 120:136, 3320:3360]
    ref = O.mlp(to_f64(x)[rows], *[to_f64(v) for v in (w1, b1, w2, b2)]) + to_f64(x)[rows]
    check_bf16("mlp in place, 3360 rows", to_f64(y)[rows], ref, noise=LAYER_NOISE, sampled=True)
    ctx.close()


# ------------------------------------------------------------------ a7-a9 attention
# Tolerances of the attention layer.  Each stage is judged on the GPU's own upstream result, so the
# stated bound (1e-2 of the RMS, or the output's own rounding floor + 2e-3) applies as it is: the
# core normalises with the sum of the very bf16 probabilities that multiply V, so their rounding
# (relative 2^-9, independent from key to key) enters as noise of 2^-9 sqrt(sum p^2 (v-o)^2) / sum p,
# far below the rounding of the output unless a single key holds the row - and then v = o.
# End to end the oracle rounds nothing while the GPU stores qkv, o and y in bf16: helpers.LAYER_NOISE
# is the allowance for that.


def score_bounds(qkv, heads=16):
    """Cauchy-Schwarz bound |q| max_k |k| on the base-2 scores of every (row, head), from the
    library's own qkv buffer (whose K carries the softmax scale): which of the kernel's two softmax
    forms a row takes depends on it."""
    m, d = qkv.shape[0], qkv.shape[1] // 3
    q = qkv[:, :d].reshape(m, heads, d // heads)
    k = qkv[:, d:2 * d].reshape(m, heads, d // heads)
    return np.sqrt((q * q).sum(-1)) * np.sqrt((k * k).sum(-1)).max(0)


FIXED_REF_LIMIT = 80.0  # the library's kFaFixedRefLimit


def shift_up(rows):  # its fa_shift_up, for values below 2^20
    return 126 - 20 - int(np.ceil(np.log2(rows)))


def shift_down(rows):  # and its fa_shift_down
    return 126 - 24 - int(np.ceil(np.log2(rows)))


@pytest.mark.parametrize("wl", [WORKLOADS["C1"], MID], ids=lambda w: w.name)
def test_global_attention(lib, wl):
    _, tok = _inputs(wl)
    _, ref = _oracle_plan(wl)
    m = ref["sizes"]["M"]
    xm = torch.from_numpy(O.merge(to_f64(tok), ref["dst_of"], m).astype(np.float32)).to(torch.bfloat16)
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(wl, 0)
    # second pass with 4x larger projection weights: the softmax becomes far from uniform
    # (random-init 0.02 weights alone give nearly flat attention, which would hide
    # indexing mistakes) and the score bound of most rows passes the limit of the
    # fixed-reference form, so the shifted form runs (and, for a few warps, the online form)
    w_big = (w_qkv.float() * 4.0).to(torch.bfloat16)
    ctx = _ctx(lib, wl)
    for tag, wq in (("stock", w_qkv), ("4x", w_big)):
        y = ctx.global_attn(xm.cuda(), wq.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
        ctx.poll()
        # each stage against the oracle fed with the GPU's own upstream (bf16) result
        ref_qkv = fold_k(O.linear(to_f64(xm), to_f64(wq), to_f64(b_qkv)))
        qkv = to_f64(ctx.debug_buffer(0))
        check_bf16(f"{wl.name}/{tag}: qkv projection", qkv, ref_qkv)
        b = score_bounds(qkv)
        report(f"{wl.name}/{tag}: score bound", max=b.max(), share_fixed_reference=float((b <= FIXED_REF_LIMIT).mean()))
        if tag == "stock":
            assert b.max() <= FIXED_REF_LIMIT  # every row takes the fixed-reference form
        else:
            forms = softmax_forms(qkv)
            assert forms["shifted"] > 0.9 * sum(forms.values())
        ref_o = O.attention_core(unfold_k(qkv), heads=16)
        o = to_f64(ctx.debug_buffer(1))
        check_bf16(f"{wl.name}/{tag}: attention core", o, ref_o, elem_noise=CORE_NOISE)
        ref_y = O.linear(o, to_f64(w_o), to_f64(b_o))
        check_bf16(f"{wl.name}/{tag}: output projection", to_f64(y), ref_y)
        if tag == "stock":  # end to end (bf16 intermediates on the GPU side, none in the oracle)
            ref_full = O.global_attention(to_f64(xm), to_f64(wq), to_f64(b_qkv), to_f64(w_o), to_f64(b_o), heads=16)
            check_bf16(f"{wl.name}: attention layer end to end", to_f64(y), ref_full, noise=LAYER_NOISE)
    ctx.close()


@pytest.mark.parametrize("grid,sharpness,form", [((22, 33), 4.0, "fixed"), ((22, 33), 6.0, "fixed"), ((22, 33), 16.0, "shifted"),
                                                 ((22, 33), 64.0, "online"), ((34, 44), 4.0, "fixed")])
def test_attention_core_with_peaked_softmax(lib, grid, sharpness, form):
    """Rows in groups of near-duplicates spread through the sequence and query weights a multiple of
    the key weights: a row's probability mass sits on itself and its group, so every key tile
    matters.  sharpness 4 and 6 keep the score bounds under the fixed-reference limit (6: up to 70, the upper
    part of what that form takes), 16 puts them over, where one shifted reference serves, 64 far over."""
    ctx = lib.LiteVGGT(2, grid[0], grid[1], 0.0)  # merge ratio 0: M = N (1462 / 3002 rows, ragged tiles)
    m = ctx.n_merged
    assert m == ctx.n_tokens
    x, w_qkv, b_qkv, w_o, b_o = make_peaked_attention_inputs(m, 31 + m, groups=97, sharpness=sharpness)
    y = ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    qkv = to_f64(ctx.debug_buffer(0))
    b = score_bounds(qkv)
    report(f"peaked m={m} s={sharpness}: score bound", max=b.max(), min=b.min())
    forms = softmax_forms(qkv)
    assert forms.get(form, 0) > 0.9 * sum(forms.values())
    qkv_o = unfold_k(qkv)
    ref_o = O.attention_core(qkv_o, heads=16)
    o = to_f64(ctx.debug_buffer(1))
    check_bf16(f"peaked m={m} s={sharpness}: attention core", o, ref_o, elem_noise=CORE_NOISE)
    # the case is what it claims to be: the rows of a query's own group hold most of its mass, so
    # leaving out the keys of one tile (planted on the oracle's side) moves the result far beyond
    # the tolerance
    keep = np.ones(m, bool)
    keep[256:384] = False
    rows = np.flatnonzero(keep)[:200]
    short = qkv_o[keep]
    ref_short = O.attention_core(short, heads=16, rows=np.arange(200))
    assert rel_err(o[rows], ref_short) > 20 * bf16_bound(ref_o)
    check_bf16(f"peaked m={m} s={sharpness}: output projection", to_f64(y), O.linear(o, to_f64(w_o), to_f64(b_o)))
    ctx.close()


# ------------------------------------------------------------------ Q/K normalisation and rotary embedding
def softmax_forms(qkv, heads=16, limit=FIXED_REF_LIMIT):
    """Which of the kernel's three softmax forms every warp of 32 rows takes, per head: "fixed" where all
    its rows have a score bound under the limit, "shifted" where bound and the maximum over the first
    64 keys leave room for one whole-number reference, else "online"."""
    m, d = qkv.shape[0], qkv.shape[1] // 3
    b = score_bounds(qkv, heads)
    forms = {}
    for h in range(heads):
        q, k = qkv[:, h * 64:h * 64 + 64], qkv[:, d + h * 64:d + h * 64 + 64]
        first = (q @ k[:64].T).max(1)
        shift = np.ceil(np.maximum(b[:, h] - shift_up(m), first)) - first <= shift_down(m)
        for w in range(0, m, 32):
            if (b[w:w + 32, h] <= limit).all():
                form = "fixed"
            else:
                form = "shifted" if shift[w:w + 32].all() else "online"
            forms[form] = forms.get(form, 0) + 1
    return forms


@pytest.mark.parametrize("frames,grid,sharpness,form", [
    (1, (1, 1), 1.0, "fixed"), (1, (1, 59), 16.0, "shifted"), (1, (2, 30), 16.0, "shifted"), (1, (3, 41), 64.0, "online"),
    (1, (2, 62), 1.0, "fixed"), (1, (11, 17), 64.0, "online"), (1, (4, 47), 64.0, "online"), (1, (14, 18), 16.0, "shifted"),
    (4, (64, 64), 1.0, "fixed"), (4, (64, 64), 16.0, "shifted"), (4, (64, 64), 64.0, "online")])
def test_attention_core_at_tile_edges_in_every_softmax_form(lib, frames, grid, sharpness, form):
    """Sequence lengths around the 64-key halves, the 128-row tiles and (16,404 rows: 129 tiles, the last
    with 20 rows and without a second half) the pairs of tiles of a CTA; there the last four of 1040 jobs,
    the rows from 15,616 on of the last head, are split along the keys and added up."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], 0.0)
    m = ctx.n_merged
    g = torch.Generator().manual_seed(77 + m)
    x = torch.randn(m, 1024, generator=g).to(torch.bfloat16)
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(WORKLOADS["C1"], 3)
    w_qkv[:1024] *= sharpness
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    qkv = to_f64(ctx.debug_buffer(0))
    assert softmax_forms(qkv).get(form, 0) > 0
    rows = np.arange(m) if m < 4096 else np.r_[0:40, 8190:8230, 15600:15632, m - 40:m]
    ref_o = O.attention_core(unfold_k(qkv), heads=16, rows=rows)
    # The probabilities are rounded to bf16, each off by at most 2^-9 relative, and the row sum is formed
    # from the rounded values: an output moves by 2^-9 sum_i d_i p_i (v_i - o), |d_i| <= 1.  Rows of random
    # keys do not average that away, so it is bounded per entry: Hoeffding's inequality for independent
    # d_i, taken where 1e7 entries together exceed it with a chance of 1e-6 (a factor sqrt(2 ln 2e13) = 7.8).
    u, worst = unfold_k(qkv), 0.0
    for h in range(16):
        q, k, v = (u[:, i * 1024 + h * 64:i * 1024 + h * 64 + 64] for i in range(3))
        s = q[rows] @ k.T / 8.0
        p = np.exp(s - s.max(1, keepdims=True))
        p2 = (p / p.sum(1, keepdims=True)) ** 2
        o = ref_o[:, h * 64:h * 64 + 64]
        worst = max(worst, float((p2 @ (v * v) - 2 * o * (p2 @ v) + o * o * p2.sum(1, keepdims=True)).max()))
    noise = 7.8 * 2.0 ** -9 * np.sqrt(worst) / float(np.sqrt(np.mean(ref_o * ref_o)))
    check_bf16(f"edges m={m} s={sharpness}: attention core", to_f64(ctx.debug_buffer(1))[rows], ref_o, noise=noise,
               sampled=m >= 4096)
    ctx.close()


def uniform_rows_ctx(lib, rows, qkv_dtype=0):
    """A context whose merged sequence is `rows` tokens without special ones, and zeroed weights for it."""
    ctx = lib.LiteVGGT(-(-rows // 4096), 64, min(64, rows // 64), 0.0, n_special=0, qkv_dtype=qkv_dtype)
    assert ctx.n_merged == rows
    zeros = [torch.zeros(*s, dtype=torch.bfloat16) for s in ((rows, 1024), (3072, 1024), (3072,), (1024, 1024), (1024,))]
    return ctx, zeros


@pytest.mark.parametrize("rows,qkv_dtype", [(4096, 0), (8192, 0)])
def test_exponentials_are_equally_good_at_every_key_position(lib, rows, qkv_dtype):
    """Some positions of a key tile take their exponential from the special-function unit (within 1.45e-7), others
    from a polynomial (within 6.6e-8, where the fixed reference does not serve).  All keys of a row score the same
    here and V is +1 at the positions 0 and -1 at the positions 31 of every 32, so an output is exactly zero
    unless the two round to different probabilities.  That takes a rounding boundary between them, within
    2.2e-7 relative where neighbours lie 2^-8 apart (bf16): 5.5e-5 of the rows, 4 or 8 of
    65,536 or 131,072, and 30 with a chance below 1e-8; a cubic (7.5e-5) splits hundreds."""
    ctx, (x, w_qkv, b_qkv, w_o, b_o) = uniform_rows_ctx(lib, rows, qkv_dtype)
    g = torch.Generator().manual_seed(rows)
    x[:, :16] = 100 + 100 * torch.rand(rows, 16, generator=g).to(torch.bfloat16)
    x[:, 16:32] = torch.randn(rows, 16, generator=g).to(torch.bfloat16)
    x[::32, 32], x[31::32, 32] = 1.0, -1.0
    for h in range(16):  # q = (x_h, x_16+h), k = (1, 1/64) before the softmax scale, v = x_32
        w_qkv[64 * h, h] = w_qkv[64 * h + 1, 16 + h] = w_qkv[2048 + 64 * h, 32] = 1.0
        b_qkv[1024 + 64 * h], b_qkv[1024 + 64 * h + 1] = 8.0, 0.125
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    assert set(softmax_forms(to_f64(ctx.debug_buffer(0)))) == {"shifted"}
    o = to_f64(ctx.debug_buffer(1))[:, ::64]
    split = int((o != 0).sum())
    report(f"probabilities that differ by position, {rows} rows, qkv_dtype {qkv_dtype}", rows=o.size, split=split)
    assert np.abs(o).max() < 2.0 ** -7 and split <= 30
    ctx.close()


def test_e4m3_probabilities_do_not_depend_on_the_key_position(lib):
    """Key 0 holds every row's maximum, all other keys score zero; V is +1 at the positions 0 and -1 at the
    positions 31 of every 32 of them, so an output is exactly zero where equal scores give equal
    probabilities.  (A cubic at some positions, 7.5e-5 off, split dozens of the 131,072 rows.)"""
    rows = 8192
    ctx, (x, w_qkv, b_qkv, w_o, b_o) = uniform_rows_ctx(lib, rows, qkv_dtype=1)
    g = torch.Generator().manual_seed(rows)
    x[:, :16] = 0.25 + 3 * torch.rand(rows, 16, generator=g).to(torch.bfloat16)
    x[:, 16:32] = torch.rand(rows, 16, generator=g).to(torch.bfloat16)
    x[32::32, 32], x[63::32, 32], x[0, 33] = 1.0, -1.0, 1.0
    for h in range(16):
        w_qkv[64 * h, h] = w_qkv[64 * h + 1, 16 + h] = w_qkv[2048 + 64 * h, 32] = 1.0
        w_qkv[1024 + 64 * h, 33], w_qkv[1024 + 64 * h + 1, 33] = 12 + h / 2, 9 - h / 4
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    o = to_f64(ctx.debug_buffer(1))[:, ::64]
    report("E4M3 probabilities that differ by position", rows=o.size, split=int((o != 0).sum()))
    assert not o.any()
    ctx.close()


@pytest.mark.parametrize("key", [128, 159])  # first and last of the 32 keys that a thread takes at a time
@pytest.mark.parametrize("rows,qkv_dtype", [(4096, 0), (8192, 0), (4096, 1)])
def test_a_key_that_is_not_a_number_shows_in_every_output(lib, rows, qkv_dtype, key):
    """One token's K of one head overflows before its normalisation and is NaN after it, with a finite V: every
    row attends to it, so that head's outputs are NaN throughout, and no other head's."""
    ctx, (x, w_qkv, b_qkv, w_o, b_o) = uniform_rows_ctx(lib, rows, qkv_dtype)
    g = torch.Generator().manual_seed(rows + key)
    x[:] = torch.randn(rows, 1024, generator=g).to(torch.bfloat16)
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(WORKLOADS["C1"], 0)
    x[:, 7], w_qkv[:, 7] = 0.0, 0.0
    x[key, 7], w_qkv[1024 + 3 * 64:1024 + 4 * 64, 7] = 2.0 ** 100, 2.0 ** 100
    one, zero = torch.ones(64, dtype=torch.bfloat16).cuda(), torch.zeros(64, dtype=torch.bfloat16).cuda()
    ctx.global_attn_ext(None, x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda(), q_norm=(10 * one, zero), k_norm=(one, zero))
    ctx.poll()
    qkv, o = ctx.debug_buffer(0).float().cpu().numpy(), ctx.debug_buffer(1).float().cpu().numpy()
    bad = np.isnan(qkv)
    assert bad[key, 1024 + 192:1024 + 256].all() and bad.sum() == 64
    if qkv_dtype == 0:
        assert set(softmax_forms(np.nan_to_num(qkv).astype(np.float64))) == {"shifted"}
    nan = np.isnan(o)
    assert nan[:, 192:256].all() and not nan[:, :192].any() and not nan[:, 256:].any()
    ctx.close()


@pytest.mark.parametrize("above", [87.0, 90.5])
def test_shifted_reference_loses_nothing_that_fp32_would_keep(lib, above):
    """Keys 0 and 1 score 0, the highest; key 1 is long, across the queries, so that the score bound lies 92 +
    `above` over it: at 87 one reference serves (16,384 rows: up to 88 binades over the highest score),
    at 90.5 the running maximum has to.  The other keys sit 40 binades down with V = 1 where keys 0 and 1 have V = 0,
    so the output is what they hold together, 2^-26, and an error of 2^-24 of the row's mass is allowed."""
    rows = 16384
    ctx, (x, w_qkv, b_qkv, w_o, b_o) = uniform_rows_ctx(lib, rows)
    x[2:, 0], x[1, 1], x[2:, 2] = -40.0 / 16 / K_FOLD, (92 + above) / 16 / K_FOLD, 1.0
    for h in range(16):
        b_qkv[64 * h] = 16.0
        w_qkv[1024 + 64 * h, 0] = w_qkv[1024 + 64 * h + 1, 1] = w_qkv[2048 + 64 * h, 2] = 1.0
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    qkv = to_f64(ctx.debug_buffer(0))
    assert set(softmax_forms(qkv)) == {"shifted" if above < 88 else "online"}
    ref = O.attention_core(unfold_k(qkv), heads=16, rows=np.arange(4))[:, ::64]
    got = to_f64(ctx.debug_buffer(1))[:, ::64]
    report(f"keys 40 binades down, bound {92 + above} up", got=float(got.max()), ref=float(ref.max()))
    assert ref.min() > 2.0 ** -28 and np.abs(got - ref[0]).max() <= 2.0 ** -24
    ctx.close()


@pytest.mark.parametrize("grid", [(1, 1), (1, 59), (4, 15), (3, 41), (4, 31)], ids=lambda g: f"{g[0]}x{g[1]}")
def test_frame_attention_at_tile_edges(lib, grid):
    """6, 64, 65, 128 and 129 tokens a frame.  The rows share a common part, as a frame's tokens do:
    LAYER_NOISE is stated against the RMS of outputs that do not average out to sigma / sqrt(rows), where
    the rounding of p (2^-9 per key, relative to sigma / sqrt(rows) too) would be of the output's own size."""
    ctx = lib.LiteVGGT(3, grid[0], grid[1], 0.5)
    n = ctx.n_tokens
    g = torch.Generator().manual_seed(5 + n)
    x = (torch.randn(1, 1024, generator=g) + 0.5 * torch.randn(n, 1024, generator=g)).to(torch.bfloat16)
    w = make_attention_weights(WORKLOADS["C1"], 4)
    y = ctx.frame_attn(x.cuda(), *[t.cuda() for t in w])
    ctx.poll()
    ref = O.frame_attention(to_f64(x), 3, *[to_f64(t) for t in w])
    check_bf16(f"frame attention, {n // 3} tokens a frame", to_f64(y), ref, noise=LAYER_NOISE)
    ctx.close()


@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD], ids=lambda w: w.name)
@pytest.mark.parametrize("mode", ["norm", "rope", "both"])
def test_global_attention_with_qk_norm_and_rope(lib, wl, mode):
    img, tok = _inputs(wl)
    ctx = _ctx(lib, wl)
    x = tok.cuda()
    plan = ctx.merge_plan(x, ctx.grad_map(img.cuda()))
    ex = ctx.plan_export(plan)
    xm = ctx.merge(plan, x)
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(wl, 0)
    gen = torch.Generator().manual_seed(wl.seed + 77)
    affine = [(1.0 + 0.2 * torch.randn(64, generator=gen)).to(torch.bfloat16) if i % 2 == 0
              else (0.2 * torch.randn(64, generator=gen)).to(torch.bfloat16) for i in range(4)]
    ext = {}
    if mode in ("norm", "both"):
        ext.update(q_gamma=to_f64(affine[0]), q_beta=to_f64(affine[1]), k_gamma=to_f64(affine[2]),
                   k_beta=to_f64(affine[3]), eps=1e-5)
    if mode in ("rope", "both"):
        # a merged row sits where the token that owns it sits
        ext.update(pos=O.token_positions(wl.frames, wl.grid_h, wl.grid_w)[ex["kept_idx"]], base=100.0)
    dev = [t.cuda() for t in affine]
    y = ctx.global_attn_ext(plan, xm, w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda(),
                            q_norm=(dev[0], dev[1]) if "q_gamma" in ext else None,
                            k_norm=(dev[2], dev[3]) if "q_gamma" in ext else None,
                            rope="pos" in ext)
    ctx.poll()
    xm64 = to_f64(xm)
    w64 = [to_f64(t) for t in (w_qkv, b_qkv, w_o, b_o)]
    # the transformed Q and K against the oracle's (two roundings on the GPU side: the projection's
    # output and the transformed values; V must be untouched)
    ref_y, ref_qkv, _ = O.global_attention(xm64, *w64, heads=16, return_parts=True, ext=ext)
    ref_qkv = fold_k(ref_qkv)
    qkv = to_f64(ctx.debug_buffer(0))
    d = 1024
    for name, sl in (("Q", slice(0, d)), ("K", slice(d, 2 * d)), ("V", slice(2 * d, 3 * d))):
        # V is one rounding from the oracle's; Q and K were rounded once by the projection and once more
        # after the transform: a second error of the size of the first, up to a quarter more in units of
        # RMS after rotating pairs in which a small entry inherits the rounding of a large partner
        second = 0.0 if name == "V" else 1.25 * rel_err(bf16_round(ref_qkv[:, sl]), ref_qkv[:, sl])
        check_bf16(f"{wl.name}/{mode}: {name}", qkv[:, sl], ref_qkv[:, sl], noise=second)
    plain = fold_k(to_f64(ctx.linear(xm, w_qkv.cuda(), b_qkv.cuda())))
    assert np.array_equal(qkv[:, 2 * d:], plain[:, 2 * d:])
    # the core on the GPU's own transformed Q/K/V, and the layer end to end
    ref_o = O.attention_core(unfold_k(qkv), heads=16)
    check_bf16(f"{wl.name}/{mode}: attention core", to_f64(ctx.debug_buffer(1)), ref_o, elem_noise=CORE_NOISE)
    # one more stored rounding than the plain layer (the transformed Q and K)
    check_bf16(f"{wl.name}/{mode}: layer end to end", to_f64(y), ref_y, noise=LAYER_NOISE)
    # and the options did something: Q is far from the plain projection
    assert rel_err(qkv[:, :d], plain[:, :d]) > 0.5
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("qkv_dtype", [0, 1])
def test_ext_entry_without_options_is_the_plain_layer(lib, qkv_dtype):
    """Neither normalisation nor rotation (and no plan): bit for bit what global_attn returns."""
    wl = WORKLOADS["C1"]
    ctx = _ctx(lib, wl, qkv_dtype=qkv_dtype)
    g = torch.Generator().manual_seed(11)
    xm = torch.randn(ctx.n_merged, 1024, generator=g).to(torch.bfloat16).cuda()
    w = [t.cuda() for t in make_attention_weights(wl, 0)]
    plain, plain_qkv = ctx.global_attn(xm, *w), ctx.debug_buffer(0)
    ext, ext_qkv = ctx.global_attn_ext(None, xm, *w), ctx.debug_buffer(0)
    ctx.poll()
    assert torch.equal(ext_qkv, plain_qkv) and torch.equal(ext, plain)
    ctx.close()


# ------------------------------------------------------------------ other sub-layers of a block
@pytest.mark.parametrize("wl", [WORKLOADS["C1"], ODD], ids=lambda w: w.name)
def test_layernorm_frame_attention_and_mlp(lib, wl):
    _, tok = _inputs(wl)
    w = make_block_weights(wl, 0)
    ctx = _ctx(lib, wl)
    x = tok.cuda()
    x64 = to_f64(tok)
    # LayerNorm: fp32 two-pass statistics, one rounding
    g, b = w["ln1"]
    xn = ctx.layernorm(x, g.cuda(), b.cuda(), eps=1e-6)
    ctx.poll()
    ref_n = O.layernorm(x64, to_f64(g), to_f64(b), 1e-6)
    check_bf16(f"{wl.name}: LayerNorm", to_f64(xn), ref_n)
    # frame-local attention on the GPU's own normalised rows, residual = the block input
    aw = [t.cuda() for t in w["attn"]]
    y = ctx.frame_attn(xn, *aw, residual=x)
    ctx.poll()
    ref_y = O.frame_attention(to_f64(xn), wl.frames, *[to_f64(t) for t in w["attn"]], heads=16, residual=x64)
    # qkv, o and y are stored in bf16 on the way, as for the global layer end to end
    check_bf16(f"{wl.name}: frame attention layer", to_f64(y), ref_y, noise=LAYER_NOISE)
    # no token may see another frame: perturbing one frame must leave the others' rows bit-identical
    x2 = xn.clone()
    t = wl.tokens_per_frame
    x2[t:2 * t] += 1.0
    y2 = ctx.frame_attn(x2, *aw, residual=x)
    ctx.poll()
    keep = torch.ones(wl.n_tokens, dtype=torch.bool, device="cuda")
    keep[t:2 * t] = False
    assert torch.equal(y[keep], y2[keep]) and not torch.equal(y[~keep], y2[~keep])
    # MLP with exact GELU; the hidden activations are stored in bf16
    mw = [t_.cuda() for t_ in w["mlp"]]
    z = ctx.mlp(xn, *mw, residual=x)
    ctx.poll()
    ref_z = O.mlp(to_f64(xn), *[to_f64(t_) for t_ in w["mlp"]], residual=x64)
    check_bf16(f"{wl.name}: MLP", to_f64(z), ref_z, noise=LAYER_NOISE)
    ctx.close()


@pytest.mark.parametrize("rows", [40, 1044])
def test_gelu_of_values_that_are_not_ordinary(lib, rows):
    """One hidden unit of the MLP takes infinities, NaN, the largest finite values and where the tails end; the
    others are zero.  The second layer hands it through, so a row is gelu(its value), rounded twice to bf16."""
    ctx = _ctx(lib, WORKLOADS["C1"])
    big = 2.0 ** 64
    hidden = [np.inf, -np.inf, np.nan, 3.0 * 2.0 ** 126, -3.0 * 2.0 ** 126, 2.0 ** 100, -2.0 ** 100, 0.0, 2.0 ** -60, -2.0 ** -60]
    hidden += [s * v for v in (0.5, 1.0, 5.5, 12.0, 13.0, 18.0, 63.5, 64.0, 64.5, 70.0, 300.0) for s in (1.0, -1.0)]
    x = torch.zeros(rows, 1024, dtype=torch.bfloat16)
    # (infinities as products that overflow)
    factor = [np.copysign(2.0 ** 65, v) if np.isinf(v) else v / big for v in hidden]
    x[:len(hidden), 0] = torch.tensor(factor, dtype=torch.float64).to(torch.bfloat16)
    w1, w2 = torch.zeros(4096, 1024, dtype=torch.bfloat16), torch.zeros(1024, 4096, dtype=torch.bfloat16)
    w1[0, 0] = big
    w2[:, 0] = 1.0
    y = ctx.mlp(x.cuda(), w1.cuda(), None, w2.cuda(), None).cpu().double().numpy()
    ctx.poll()
    for r, v in enumerate(hidden):
        if np.isnan(v):
            assert np.isnan(y[r]).all()
        elif np.isinf(v):
            assert (y[r] == max(v, 0.0)).all()  # the limits
        else:  # two roundings to bf16, and the rational approximation's 1.5e-7 of |v| / 2 where its tail is not zero
            ref = float(O.gelu(np.array([v]))[0])
            bound = 2.0 ** -7 * abs(ref) + (0.75e-7 * abs(v) if abs(v) < 64.0 else 0.0) + 2.0 ** -133
            assert np.abs(y[r] - ref).max() <= bound, (v, ref, y[r][0])
    assert (y[len(hidden):] == 0.0).all()
    ctx.close()


# ------------------------------------------------------------------ whole layer
def test_whole_layer_c1_and_host_entry(lib):
    wl = WORKLOADS["C1"]
    img, tok = _inputs(wl)
    ctx = _ctx(lib, wl)
    x = tok.cuda()
    grad = ctx.grad_map(img.cuda())
    plan = ctx.merge_plan(x, grad)
    w = [t.cuda() for t in make_attention_weights(wl, 0)]
    xm = ctx.merge(plan, x)
    ym = ctx.global_attn(xm, *w)
    out = ctx.unmerge(plan, ym, x)
    ctx.poll()
    ex = ctx.plan_export(plan)
    x64 = to_f64(tok)
    ref_m = O.merge(x64, ex["dst_of"], ctx.n_merged)
    ref_y = O.global_attention(ref_m, *[to_f64(t) for t in w], heads=16)
    ref_out = O.unmerge(ref_y, ex["dst_of"], x64)
    # the oracle is fed the GPU's plan but none of its intermediates; the residual dominates the
    # output's scale, so the layer's stored intermediates stay inside the single-rounding bound
    # (stated bound as it is; entry by entry the attention branch's stored intermediates show: its
    # RMS is about half the output's, so half of LAYER_NOISE)
    check_bf16("C1: whole layer (merge, attention, unmerge + residual)", to_f64(out), ref_out, elem_noise=LAYER_NOISE / 2)
    x_host = tok.clone().pin_memory()
    out_host = torch.empty_like(x_host).pin_memory()
    ctx.global_layer_host(plan, x_host, *w, out_host)
    ctx.poll()
    assert torch.equal(out_host, out.cpu())
    out_host.zero_()
    plan2 = ctx.global_layer_host(None, x_host, *w, out_host, grad=grad)  # builds its own plan
    ctx.poll()
    assert torch.equal(out_host, out.cpu())
    plan2.destroy()
    times = ctx.timers_read()
    assert times["attention"][1] >= 2 and times["attention"][0] > 0.0
    assert ctx.launch_count() > 10
    plan.destroy()
    ctx.close()


@pytest.mark.parametrize("wl", [WORKLOADS["C1"], MID], ids=lambda w: w.name)
def test_pipelined_host_entry_equals_the_ordered_one(lib, wl):
    """Five independent calls in a row through the entry point whose copies run on their own streams:
    each output must be bit-identical to the ordered entry point's on the same input (the kernels are
    the same; only the copies moved), with the plan refreshed inside the third call."""
    img, tok = _inputs(wl)
    ctx = _ctx(lib, wl)
    grad = ctx.grad_map(img.cuda())
    w = [t.cuda() for t in make_attention_weights(wl, 0)]
    gen = torch.Generator().manual_seed(wl.seed + 5)
    inputs = [tok.clone().pin_memory()]
    for _ in range(4):
        inputs.append((tok.float() + 0.05 * torch.randn(tok.shape, generator=gen)).to(torch.bfloat16).pin_memory())
    # ordered entry point: one call, one synchronisation at a time
    expected, plan = [], None
    for i, xh in enumerate(inputs):
        oh = torch.empty_like(xh).pin_memory()
        plan = ctx.global_layer_host(plan, xh, *w, oh, grad=grad if i in (0, 2) else None)
        ctx.poll()
        expected.append(oh.clone())
    plan.destroy()
    outs = [torch.zeros_like(xh).pin_memory() for xh in inputs]
    plan = None
    for i, (xh, oh) in enumerate(zip(inputs, outs)):
        plan = ctx.global_layer_host_pipelined(plan, xh, *w, oh, grad=grad if i in (0, 2) else None)
    ctx.host_drain()
    ctx.poll()
    for i, (got, ref) in enumerate(zip(outs, expected)):
        assert torch.equal(got, ref), f"call {i}"
    # a second round reuses both staging slots
    for xh, oh in zip(inputs[:3], outs[:3]):
        oh.zero_()
        ctx.global_layer_host_pipelined(plan, xh, *w, oh)
    ctx.host_drain()
    ctx.poll()
    for i, xh in enumerate(inputs[:3]):
        oh = torch.empty_like(xh).pin_memory()
        ctx.global_layer_host(plan, xh, *w, oh)
        ctx.poll()
        assert torch.equal(outs[i], oh), f"second round, call {i}"
    plan.destroy()
    ctx.close()


# ------------------------------------------------------------------ bounded waits
def test_a_wait_that_runs_out_sets_the_status_word_and_leaves_the_context_usable(lib):
    """Every pipelined kernel waits on its barriers with a cycle limit.  The self-test kernel waits,
    through the same device helpers, on a barrier that nobody arrives on (limit: a million cycles,
    half a millisecond): it must return, the status poll must report the timeout once and be clean
    afterwards, and ordinary work on the same context must still be right."""
    wl = WORKLOADS["C1"]
    ctx = _ctx(lib, wl)
    a = torch.randn(300, 128, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16)
    w = (0.05 * torch.randn(320, 128, generator=torch.Generator().manual_seed(4))).to(torch.bfloat16)
    ref = to_f64(a) @ to_f64(w).T
    before = ctx.linear(a.cuda(), w.cuda(), None)
    ctx.poll()
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    outcome = ctx.selftest_bounded_wait(1_000_000)
    t1.record()
    torch.cuda.synchronize()
    assert outcome == 4, f"outcome word {outcome}: bit 2 = ran to its end, bits 0/1 = a wait reported a false completion"
    assert t0.elapsed_time(t1) < 100.0  # a million cycles, not the production limit of 2^32
    with pytest.raises(lib.LiteVGGTError) as e:
        ctx.poll()
    assert e.value.code == 9  # LITEVGGT_ERR_DEVICE_TIMEOUT
    ctx.poll()  # the flag was cleared by the poll that reported it
    after = ctx.linear(a.cuda(), w.cuda(), None)
    ctx.poll()
    assert torch.equal(before, after)
    check_bf16("linear after a timed-out wait", to_f64(after), ref)
    # limits outside [1e3, 2^32] are refused on the host
    assert ctx.lib.litevggt_selftest_bounded_wait(ctx.handle, 10, None, None) == 3
    ctx.close()


# ------------------------------------------------------------------ ABI misuse
def test_abi_misuse_returns_error_codes(lib):
    wl = WORKLOADS["C1"]
    _, tok = _inputs(wl)
    ctx = _ctx(lib, wl)
    other = lib.LiteVGGT(wl.frames, wl.grid_h, wl.grid_w, 0.25)
    # shapes the kernels are not laid out for are refused when the context is made
    for bad in (dict(patch_px=31), dict(grid_w=65)):
        kw = dict(frames=wl.frames, grid_h=wl.grid_h, grid_w=wl.grid_w)
        over = {k: v for k, v in bad.items() if k not in kw}
        kw.update({k: v for k, v in bad.items() if k in kw})
        with pytest.raises(lib.LiteVGGTError) as e:
            lib.LiteVGGT(kw["frames"], kw["grid_h"], kw["grid_w"], 0.5, **over)
        assert e.value.code == 2
    x = tok.cuda()
    _, ref = _oracle_plan(wl)
    plan = ctx.plan_import(ref["dst_of"])
    with pytest.raises(lib.LiteVGGTError) as e:
        other.merge(plan, x, torch.empty(other.n_merged, 1024, dtype=torch.bfloat16, device="cuda"))
    assert e.value.code == 8  # stale / foreign plan
    with pytest.raises(lib.LiteVGGTError) as e:
        lib.binding._check(ctx.lib.litevggt_global_attn(ctx.handle, x.data_ptr(), 17, x.data_ptr(), None,
                                                        x.data_ptr(), None, x.data_ptr(), None), "global_attn")
    assert e.value.code == 3  # shape
    with pytest.raises(lib.LiteVGGTError) as e:
        lib.binding._check(ctx.lib.litevggt_merge(ctx.handle, plan.handle, x.data_ptr() + 2, x.data_ptr(), None), "merge")
    assert e.value.code == 4  # alignment
    bad = ref["dst_of"].copy()
    bad[0] = ctx.n_merged + 5
    with pytest.raises(lib.LiteVGGTError) as e:
        ctx.plan_import(bad)
    assert e.value.code == 3
    # the block sub-layers validate their arguments too
    rc = ctx.lib.litevggt_layernorm(ctx.handle, x.data_ptr(), 16, x.data_ptr(), x.data_ptr(), 0.0, x.data_ptr(), None)
    assert rc == 3  # eps must be positive
    rc = ctx.lib.litevggt_mlp(ctx.handle, x.data_ptr(), ctx.n_tokens + 1, x.data_ptr(), None, x.data_ptr(), None, None,
                              x.data_ptr(), None)
    assert rc == 3  # more rows than the context was sized for
    rc = ctx.lib.litevggt_frame_attn(ctx.handle, x.data_ptr(), None, None, x.data_ptr(), None, None, x.data_ptr(), None)
    assert rc == 1  # missing weights
    # the extended attention layer: options struct required, the four affine vectors come together,
    # the rotation needs the plan for its positions
    import ctypes as C
    xm_ = torch.zeros(ctx.n_merged, 1024, dtype=torch.bfloat16, device="cuda")
    wq_ = torch.zeros(3072, 1024, dtype=torch.bfloat16, device="cuda")
    args = lambda plan_h, ext_ref: (ctx.handle, plan_h, xm_.data_ptr(), ctx.n_merged, wq_.data_ptr(), None,
                                    wq_.data_ptr(), None, ext_ref, xm_.data_ptr(), None)
    assert ctx.lib.litevggt_global_attn_ext(*args(None, None)) == 1
    opt = lib.binding.AttnExt()
    opt.q_norm_gamma = xm_.data_ptr()
    opt.norm_eps = 1e-5
    assert ctx.lib.litevggt_global_attn_ext(*args(None, C.byref(opt))) == 1
    opt = lib.binding.AttnExt()
    opt.rope, opt.rope_base = 1, 100.0
    assert ctx.lib.litevggt_global_attn_ext(*args(None, C.byref(opt))) == 1
    opt.rope_base = 1.0
    assert ctx.lib.litevggt_global_attn_ext(*args(plan.handle, C.byref(opt))) == 3
    # a caller partition with wrong class counts is flagged, not followed out of bounds
    cls_bad = torch.from_numpy(ref["cls"].copy())
    cls_bad[wl.tokens_per_frame + 7] = O.CLS_PROTECTED if cls_bad[wl.tokens_per_frame + 7] != O.CLS_PROTECTED else O.CLS_SRC
    p2 = ctx.merge_plan_with_partition(x, cls_bad.cuda())
    with pytest.raises(lib.LiteVGGTError) as e:
        ctx.poll()
    assert e.value.code == 10
    ctx.poll()  # flag was cleared
    p2.destroy(); plan.destroy()
    other.close(); ctx.close()


# ------------------------------------------------------------------ E4M3 variant of the attention operands
# Tolerances of the FP8 variant.  The quantised operands are judged bit for bit against the
# oracle's quantiser (same scales, same codes).  The attention core is then judged on the GPU's own
# quantised operands, dequantised, so that what remains is (a) the rounding of the probabilities to
# E4M3 - relative error up to 2^-4, independent from key to key, over the sum of the same rounded
# values: sum_i d_i p_i (v_i - o) / sum_i p_i with |d_i| <= 2^-4, i.e. at most 6.25 % of the spread
# of the values a row attends to and 1/sqrt(3 n_eff) of that when n_eff keys share the mass - and
# (b) the bf16 rounding of the output.  Nearly uniform rows (stock weights) therefore meet the bf16
# bound plus FP8_FLAT_NOISE; rows held by a handful of keys get FP8_PEAKED_NOISE.
FP8_FLAT_NOISE = 8e-3
FP8_PEAKED_NOISE = 8e-2


def _e4m3_decode(codes):
    vals = np.concatenate([O.e4m3_values(), [np.nan]])
    c = codes.cpu().numpy()
    return np.where(c & 0x80, -1.0, 1.0) * vals[c & 0x7f]


@pytest.mark.parametrize("wl", [WORKLOADS["C1"], MID], ids=lambda w: w.name)
def test_fp8_attention_variant(lib, wl):
    _, tok = _inputs(wl)
    _, ref = _oracle_plan(wl)
    m = ref["sizes"]["M"]
    xm = torch.from_numpy(O.merge(to_f64(tok), ref["dst_of"], m).astype(np.float32)).to(torch.bfloat16)
    w_qkv, b_qkv, w_o, b_o = make_attention_weights(wl, 0)
    w_big = (w_qkv.float() * 3.0).to(torch.bfloat16)
    ctx = _ctx(lib, wl, qkv_dtype=1)
    for tag, wq, noise in (("stock", w_qkv, FP8_FLAT_NOISE), ("3x", w_big, FP8_PEAKED_NOISE)):
        y = ctx.global_attn(xm.cuda(), wq.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
        ctx.poll()
        qkv = to_f64(ctx.debug_buffer(0))   # the bf16 projection, as the bf16 path produces it
        f8 = ctx.debug_fp8_buffers()
        # quantisation: scales and codes equal the oracle's on the GPU's own projection
        deq_ref, codes_ref, scales_ref = O.quantize_qkv_e4m3(qkv, heads=16)
        amax = f8["amax"].cpu().numpy()
        assert np.array_equal(amax / np.float32(448.0), scales_ref), "per-head scales"
        d = 1024
        got_codes = np.concatenate([f8["q8"].cpu().numpy(), f8["k8"].cpu().numpy(),
                                    f8["v8t"].cpu().numpy()[:, :m].T], axis=1)
        nonzero = (codes_ref & 0x7f) != 0  # the sign bit of a zero is free
        assert np.array_equal(got_codes[nonzero], codes_ref[nonzero]) and np.all((got_codes[~nonzero] & 0x7f) == 0)
        assert np.all(f8["v8t"].cpu().numpy()[:, m:] == 0), "padded keys must be zero"
        # the core on the dequantised operands
        ref_o = O.attention_core(unfold_k(deq_ref), heads=16)
        o = to_f64(ctx.debug_buffer(1))
        check_bf16(f"fp8 {wl.name}/{tag}: attention core", o, ref_o, noise=noise)
        # against the unquantised core: what the 8-bit operands cost (reported, loosely bounded)
        ref_o_bf16 = O.attention_core(unfold_k(qkv), heads=16)
        report(f"fp8 {wl.name}/{tag}: attention core vs unquantised operands", err_over_rms=rel_err(o, ref_o_bf16))
        assert rel_err(o, ref_o_bf16) < (0.1 if tag == "stock" else 1.0)
        check_bf16(f"fp8 {wl.name}/{tag}: output projection", to_f64(y), O.linear(o, to_f64(w_o), to_f64(b_o)))
    ctx.close()


def test_fp8_attention_variant_with_peaked_softmax(lib):
    """The E4M3 variant on the near-duplicate groups: every key tile matters, and a dropped tile on
    the oracle's side is far outside the FP8 tolerance too."""
    ctx = lib.LiteVGGT(2, 22, 33, 0.0, qkv_dtype=1)
    m = ctx.n_merged
    x, w_qkv, b_qkv, w_o, b_o = make_peaked_attention_inputs(m, 31 + m, groups=97, sharpness=4.0)
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    deq, _, _ = O.quantize_qkv_e4m3(to_f64(ctx.debug_buffer(0)), heads=16)
    deq = unfold_k(deq)
    ref_o = O.attention_core(deq, heads=16)
    o = to_f64(ctx.debug_buffer(1))
    check_bf16("fp8 peaked: attention core", o, ref_o, noise=FP8_PEAKED_NOISE)
    keep = np.ones(m, bool)
    keep[256:384] = False
    rows = np.flatnonzero(keep)[:200]
    ref_short = O.attention_core(deq[keep], heads=16, rows=np.arange(200))
    assert rel_err(o[rows], ref_short) > 4 * (bf16_bound(ref_o) + FP8_PEAKED_NOISE)
    ctx.close()


@pytest.mark.parametrize("frames,grid", [(1, (1, 1)), (1, (1, 59)), (1, (4, 15)), (1, (3, 41)), (1, (4, 31)), (1, (4, 47)),
                                         (1, (14, 18)), (4, (64, 64))], ids=lambda v: str(v).replace(" ", ""))
def test_fp8_attention_at_tile_edges(lib, frames, grid):
    """6 to 257 rows: one and several key tiles, ragged halves, the reference handed from one warp of a
    pair to the other after every step; 16,404 rows: the last four of 1040 jobs split along the keys.
    Rows in groups of near-duplicates, so row maxima sit anywhere in the sequence and the reference
    keeps growing."""
    ctx = lib.LiteVGGT(frames, grid[0], grid[1], 0.0, qkv_dtype=1)
    m = ctx.n_merged
    x, w_qkv, b_qkv, w_o, b_o = make_peaked_attention_inputs(m, 57 + m, groups=max(3, m // 5), sharpness=4.0)
    ctx.global_attn(x.cuda(), w_qkv.cuda(), b_qkv.cuda(), w_o.cuda(), b_o.cuda())
    ctx.poll()
    deq, _, _ = O.quantize_qkv_e4m3(to_f64(ctx.debug_buffer(0)), heads=16)
    rows = np.arange(m) if m < 4096 else np.r_[0:40, m - 800:m - 760, m - 40:m]
    ref_o = O.attention_core(unfold_k(deq), heads=16, rows=rows)
    check_bf16(f"fp8 edges m={m}: attention core", to_f64(ctx.debug_buffer(1))[rows], ref_o, noise=FP8_PEAKED_NOISE,
               sampled=m >= 4096)
    ctx.close()
