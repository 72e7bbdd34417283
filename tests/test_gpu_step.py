"""Whole-step parity: fv_var_step through the C ABI against the CPU oracle on the same seeded inputs.

Forced-index mode (the oracle's kept indices are fed to the GPU) isolates floating-point parity:
every token must be within max-abs 3e-2 and cosine >= 0.999 of the fp64 oracle.  Free-running mode
checks the integer side: the first pruned sublayer sees identical inputs on both sides, so its kept
set must match the oracle's (up to near-ties at the threshold)."""
import copy

import numpy as np
import pytest
import torch

from oracle import fastvar_oracle as O
from paper_2503_23367_b200 import binding as fv
from paper_2503_23367_b200 import inputs as I
from tests.helpers import SUB_NAMES, make_oracle, per_token_errors, run_oracle, trace_to_index_tensor
from tests.helpers import oracle_weights as helpers_oracle_weights

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MAX_ABS, MIN_COS = 3e-2, 0.999


def make_ctx(wl: I.Workload, mt: I.ModelTensors, unpruned=False, granularity=0, resid_dtype=0) -> fv.FvContext:
    cap = sum(wl.tokens(i) if (unpruned or wl.keep[i] >= 1.0) else O.kept_count(wl.keep[i], wl.sides[i], wl.sides[i])
              for i in range(len(wl.sides)))
    return fv.FvContext(wl.L, wl.C, wl.H, [(s, s) for s in wl.sides], wl.cache_step, wl.B, cap, mt,
                        cross_len=wl.cross_len, mlp_ratio=wl.mlp_ratio, device=DEV, granularity=granularity, resid_dtype=resid_dtype)


def gpu_schedule(ctx, wl, xs, forced=None, trace=False):
    outs, traces = [], []
    ctx.reset()
    for i, x in enumerate(xs):
        xd = torch.from_numpy(x).to(DEV)
        f = t = None
        if wl.keep[i] < 1.0:
            k = O.kept_count(wl.keep[i], wl.sides[i], wl.sides[i])
            if forced is not None:
                f = torch.from_numpy(forced[i]).to(DEV)
            if trace:
                t = torch.zeros((wl.L, wl.n_sub, wl.B, k), dtype=torch.int32, device=DEV)
        outs.append(ctx.var_step(xd, i, wl.keep[i], forced_idx=f, idx_trace=t).cpu().numpy())
        traces.append(None if t is None else t.cpu().numpy())
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    return outs, traces


def check_forced(wl, kind="iid"):
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i, kind) for i in range(len(wl.sides))]
    orc, ref, tr = run_oracle(wl, mt, xs)
    forced = [trace_to_index_tensor(wl, tr[i]) if wl.keep[i] < 1.0 else None for i in range(len(xs))]
    ctx = make_ctx(wl, mt)
    got, _ = gpu_schedule(ctx, wl, xs, forced=forced)
    worst = (0.0, 1.0)
    for i in range(len(xs)):
        err, cos = per_token_errors(got[i], ref[i])
        worst = (max(worst[0], err), min(worst[1], cos))
        assert err <= MAX_ABS and cos >= MIN_COS, f"step {i} side {wl.sides[i]}: max-abs {err:.4g}, cos {cos:.6f}"
    assert ctx.state() == (len(xs), orc.kv_len)
    ctx.close()
    return worst


def test_tiny_full_schedule_forced_indices():
    check_forced(I.WORKLOADS["tiny"])


def test_tiny_full_schedule_structured_maps():
    check_forced(I.WORKLOADS["tiny"], kind="structured")


def test_var_d16_shape_two_blocks_forced_indices():
    wl = I.WORKLOADS["var_d16_256"].with_depth(2)
    wl = I.Workload(wl.name, L=2, C=wl.C, H=wl.H, B=2, sides=wl.sides, keep=wl.keep, seed=wl.seed)
    check_forced(wl)


def test_var_d30_shape_one_block_forced_indices():
    base = I.WORKLOADS["var_d30_512"]
    sides = (1, 2, 4, 9, 13, 18, 24)
    wl = I.Workload("d30-short", L=1, C=base.C, H=base.H, B=2, sides=sides,
                    keep=(1.0, 1.0, 1.0, 1.0, 1.0, 0.75, 0.5), seed=base.seed)
    check_forced(wl)


def test_infinity_shape_cross_attention_forced_indices():
    base = I.WORKLOADS["infinity_2b_1k"]
    sides = (1, 2, 4, 8, 12, 16, 24)
    wl = I.Workload("inf-short", L=1, C=base.C, H=base.H, B=2, sides=sides,
                    keep=(1.0, 1.0, 1.0, 1.0, 1.0, 0.6, 0.4), cross_len=64, seed=base.seed)
    check_forced(wl)


def _bf16_t(bits):
    return torch.from_numpy(bits.view(np.int16)).to(DEV).view(torch.bfloat16)


FULL_SIZE = [("infinity_2b_1k", 820, 4403), ("infinity_2b_2k", 3277, 10369)]


@pytest.mark.parametrize("workload,k_expect,kv_expect", FULL_SIZE)
def test_full_size_last_pruned_step_of_the_bench_workload(workload, k_expect, kv_expect):
    """The last pruned step of the two Infinity-shaped workloads at FULL width and batch -- 64x64 with B 2 (820 kept
    rows per image, 4403 cached keys) and the 2K zero-shot step 128x128 with B 1 (3277 kept rows, 10369 cached keys,
    restored from the 48x48 caches); C 2048, 16 heads of 128, 512 text tokens: the shapes and launch
    configuration bench.py times -- on one transformer block (depth only repeats the same launches).
    The KV prefix of the earlier scales and the sublayer caches are seeded bf16 values placed on both
    sides.  Every output row is compared, not a sample: forced-index mode for the floating point, and
    the first selection (identical input on both sides) for the indices."""
    wl = I.WORKLOADS[workload].with_depth(1)
    step = len(wl.sides) - 1
    side = wl.sides[step]
    kv_before = sum(O.kept_count(wl.keep[i], wl.sides[i], wl.sides[i]) if wl.keep[i] < 1 else wl.tokens(i) for i in range(step))
    n_c = wl.tokens(wl.cache_step)
    mt = I.model_tensors(wl)
    x = I.step_input(wl, step, "structured")
    kpre = I.normal_bf16(wl.seed + 900, (wl.B, kv_before, wl.C))
    vpre = I.normal_bf16(wl.seed + 950, (wl.B, kv_before, wl.C))
    caches = {name: I.normal_bf16(wl.seed + 990 + j, (wl.B, n_c, wl.C), 0.5) for j, name in enumerate(SUB_NAMES[wl.n_sub])}
    widen = lambda bits: I.bf16_bits_to_f32(bits).astype(np.float64)
    # ---- oracle
    orc = make_oracle(wl, mt)
    orc.step, orc.kv_len = step, kv_before
    orc.Kc[0] = [widen(kpre[b]) for b in range(wl.B)]
    orc.Vc[0] = [widen(vpre[b]) for b in range(wl.B)]
    orc.cache[0] = {name: widen(c) for name, c in caches.items()}
    tr = {}
    ref = orc.var_step(x, step, wl.keep[step], trace=tr)
    k = O.kept_count(wl.keep[step], side, side)
    assert k == k_expect and kv_before == kv_expect and orc.kv_len == kv_before + k
    # ---- CUDA path, oracle's indices forced
    ctx = make_ctx(wl, mt)

    def place_state():
        kview, vview = ctx.kv_views(0)
        kview[:, :kv_before].copy_(_bf16_t(kpre))
        vview[:, :, :kv_before].copy_(_bf16_t(np.ascontiguousarray(vpre.transpose(0, 2, 1))))
        for si, name in enumerate(SUB_NAMES[wl.n_sub]):
            ctx.cache_view(0, si).copy_(_bf16_t(caches[name]))
        ctx.set_state(step, kv_before)
        ctx.prepare_text(wl.B)

    place_state()
    forced = torch.from_numpy(trace_to_index_tensor(wl, tr)).to(DEV)
    xd = torch.from_numpy(x).to(DEV)
    got = ctx.var_step(xd, step, wl.keep[step], forced_idx=forced).cpu().numpy()
    assert ctx.device_status() == 0 and ctx.state() == (step + 1, kv_before + k)
    err, cos = per_token_errors(got, ref)
    assert err <= MAX_ABS and cos >= MIN_COS, (err, cos)
    # rows that were not forwarded anywhere in the block only ever received restored cache rows
    # ---- free running: the first selection sees the same x on both sides
    place_state()
    trace = torch.zeros((wl.L, wl.n_sub, wl.B, k), dtype=torch.int32, device=DEV)
    ctx.var_step(xd, step, wl.keep[step], idx_trace=trace)
    assert ctx.device_status() == 0
    idx_g = trace[0, 0].cpu().numpy().astype(np.int64)
    idx_o, s_o = tr[(0, "attn")]["idx"], tr[(0, "attn")]["score"]
    for b in range(wl.B):
        assert np.all(np.diff(idx_g[b]) > 0)
        diff = np.setxor1d(idx_g[b], idx_o[b])
        if len(diff):
            tau = np.sort(s_o[b])[::-1][k - 1]
            assert np.all(np.abs(s_o[b, diff] - tau) <= 1e-5 * tau), "index mismatch away from a near-tie"
    # the later selections read the column sums the restorations left behind; their inputs differ from the oracle's by
    # the bf16 rounding of the branch before them, so on this structured map (bimodal scores) the sets must be valid and
    # agree with the oracle's free-running ones on all but the tokens next to the threshold
    for si, name in enumerate(SUB_NAMES[wl.n_sub]):
        g = trace[0, si].cpu().numpy().astype(np.int64)
        for b in range(wl.B):
            assert np.all(np.diff(g[b]) > 0) and g[b, 0] >= 0 and g[b, -1] < side * side
            overlap = len(np.intersect1d(g[b], tr[(0, name)]["idx"][b])) / k
            assert overlap >= 0.98, (name, b, overlap)
    ctx.close()


def _zero_branch_tensors(wl):
    """Model tensors whose sublayer branches all end in a zero projection (w_o, b_o, w_o_x, w_fc2, b_fc2 = 0):
    every branch output y is exactly 0 on both sides, whatever the bf16 path computes before it."""
    mt = I.model_tensors(wl)
    for lst in (mt.w_o, mt.b_o, mt.w_o_x, mt.w_fc2, mt.b_fc2):
        for a in lst:
            a[...] = 0
    return mt


ZERO_BRANCH_CASES = [  # h, w, hc, wc, C, H, B, B_max, keep, kind, oracle_runs_the_step
    (40, 40, 32, 32, 2048, 16, 2, 2, 0.6, "structured", False),      # 128 kept rows or more: the last GEMM leaves their sums, the side stream one
    (48, 48, 32, 32, 2048, 16, 2, 2, 0.4, "structured", False),      # partial of all the others (fused: groups of chunks, folded through global memory)
    (64, 64, 32, 32, 2048, 16, 2, 2, 0.2, "structured", False),
    (64, 64, 32, 32, 2048, 16, 2, 2, 0.2, "iid", False),
    (33, 31, 10, 10, 256, 4, 3, 4, 0.5, "iid", True),                # ragged last chunk, partial batch
    (50, 50, 13, 13, 1920, 30, 1, 1, 0.25, "structured", True),
    (96, 96, 48, 48, 2048, 16, 1, 1, 0.2, "structured", False),
    (128, 128, 48, 48, 2048, 16, 1, 1, 0.2, "structured", False),    # the 2K zero-shot step
]
# Fewer than 128 kept rows: a launch of its own restores them and folds the chunks of all rows, group by group.
ZERO_BRANCH_FEW_ROWS = [
    (33, 31, 10, 10, 256, 4, 3, 4, 0.12, "iid", True),               # groups of 2, ragged last chunk, partial batch
    (40, 40, 32, 32, 2048, 16, 2, 2, 0.07, "structured", False),     # groups of 4, each folded by a cluster
    (48, 48, 32, 32, 2048, 16, 2, 2, 0.05, "structured", False),     # 5
    (64, 64, 32, 32, 2048, 16, 2, 2, 0.03, "structured", False),     # 8
    (50, 50, 13, 13, 1920, 30, 1, 1, 0.05, "structured", False),     # ragged last group (79 chunks in groups of 5)
    (96, 96, 48, 48, 2048, 16, 1, 1, 0.0135, "structured", False),   # 18: through global memory
    (128, 128, 48, 48, 2048, 16, 1, 1, 0.0077, "structured", False), # 32
]


@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("h,w,hc,wc,C,H,B,B_max,keep,kind,full_oracle", ZERO_BRANCH_CASES)
def test_every_selection_of_a_step_on_bit_identical_input(h, w, hc, wc, C, H, B, B_max, keep, kind, full_oracle, fused):
    """Inside fv_var_step only the first selection sums the token map itself; every later one takes Eq. 4's column
    sums from the restoration before it (rows that were not kept on a side stream, kept rows by the last
    GEMM).  With every branch ending in a zero projection and zero sublayer caches, each restoration adds exactly 0,
    so x entering EVERY sublayer is bit-identical on both sides and each of the 2 blocks x 3 selections must keep
    the oracle's set (any difference on a near-tie at the threshold, within 1e-5 relative).  Runs at the bench
    shapes' maps, at ragged chunk / group counts and with a partial batch, in both forms the step has: the separate
    kernels (the default) and one fused launch per selection (kept rows of the previous sublayer restored and
    summed inside it, grid-wide wait, gather of the new rows)."""
    if full_oracle and fused:
        full_oracle = False          # the oracle's own step is run once, in the default form
    wl = I.Workload("zero-branch", L=2, C=C, H=H, B=B_max, sides=(hc, h), keep=(1.0, keep), cross_len=64, mlp_ratio=1, seed=811)
    mt = _zero_branch_tensors(wl)
    n, k = h * w, O.kept_count(keep, h, w)
    x = I.token_map(900 + h, B, h, w, C, kind)
    ctx = fv.FvContext(wl.L, C, H, [(hc, wc), (h, w)], 0, B_max, k, mt, cross_len=64, mlp_ratio=1, device=DEV)
    for l in range(wl.L):
        for si in range(3):
            ctx.cache_view(l, si).zero_()
    ctx.set_state(1, 0)
    ctx.prepare_text(B)
    trace = torch.full((wl.L, 3, B, k), -1, dtype=torch.int32, device=DEV)
    xd = torch.from_numpy(x).to(DEV)
    assert fv.lib().fv_step_fused_selection(fused) == 0
    try:
        got = ctx.var_step(xd, 1, keep, idx_trace=trace).cpu().numpy()
    finally:
        fv.lib().fv_step_fused_selection(0)
    assert ctx.device_status() == 0 and ctx.state() == (2, k)
    assert np.array_equal(got, x), "a zero branch changed the residual stream"
    # the oracle's selection of this (unchanged) map: one score vector serves all six sublayers
    score_o = O.pts_score(x)
    idx_o = O.pts_topk(score_o, k)
    if full_oracle:     # small enough to run the oracle's whole step: it must agree that nothing changes
        w64 = helpers_oracle_weights(mt)
        w64 = dict(w64); w64["mod"] = w64["mod"][:, :B]; w64["text"] = w64["text"][:B]
        orc = O.VarOracle(wl.L, C, H, [(hc, wc), (h, w)], cache_step=0, weights=w64, B=B, cross_len=64)
        orc.step, orc.kv_len = 1, 0
        for l in range(wl.L):
            orc.cache[l] = {name: np.zeros((B, hc * wc, C)) for name in SUB_NAMES[3]}
        tr = {}
        ref = orc.var_step(x, 1, keep, trace=tr)
        assert np.array_equal(ref, x.astype(np.float64))
        for l in range(wl.L):
            for name in SUB_NAMES[3]:
                assert np.array_equal(tr[(l, name)]["idx"], idx_o)
    idx_g = trace.cpu().numpy().astype(np.int64)
    tau = np.sort(score_o, axis=1)[:, ::-1][:, k - 1]
    flips = 0
    for l in range(wl.L):
        for si in range(3):
            for b in range(B):
                g = idx_g[l, si, b]
                assert np.all(np.diff(g) > 0) and g[0] >= 0 and g[-1] < n, (l, si, b)
                diff = np.setxor1d(g, idx_o[b])
                flips += len(diff)
                assert np.all(np.abs(score_o[b, diff] - tau[b]) <= 1e-5 * tau[b]), f"block {l} sublayer {si} image {b}: kept set differs away from a near-tie"
    assert flips <= max(4, 6 * B * k // 100), f"{flips} near-tie flips: the near-tie rule is carrying the test"
    ctx.close()


@pytest.mark.parametrize("h,w,hc,wc,C,H,B,B_max,keep,kind,full_oracle", ZERO_BRANCH_FEW_ROWS)
def test_every_selection_of_a_step_that_keeps_few_rows(h, w, hc, wc, C, H, B, B_max, keep, kind, full_oracle):
    assert O.kept_count(keep, h, w) < 128
    test_every_selection_of_a_step_on_bit_identical_input(h, w, hc, wc, C, H, B, B_max, keep, kind, full_oracle, 0)


# Maps small enough for the one-launch form (a cluster of CTAs per image): one row per CTA, CTAs without a row, ragged last CTA, clusters
# of 16 and (eight images) of 8, one and two chunks of rows per thread, channel groups that are not whole warps.  Those that keep 128 rows or more on more
# than a few rows per CTA go with the last GEMM instead (18 x 18 at 0.75, 20 x 28 at 0.9: test_route_of_a_pruned_step has both).
SMALL_MAPS = [(1, 3, 1, 1, 128, 2, 2, 2, 0.5, "iid"), (5, 7, 3, 3, 256, 4, 3, 4, 0.3, "iid"), (16, 16, 10, 10, 1024, 16, 1, 1, 0.5, "structured"),
              (13, 13, 10, 10, 1024, 16, 8, 8, 0.6, "structured"), (18, 18, 13, 13, 1920, 30, 2, 3, 0.75, "structured"), (24, 24, 9, 13, 256, 4, 2, 2, 0.15, "iid"),
              (12, 12, 8, 8, 2048, 16, 2, 2, 0.6, "structured"), (20, 28, 13, 13, 384, 6, 1, 1, 0.9, "iid"),
              (18, 18, 13, 13, 1920, 30, 2, 3, 0.35, "structured"), (20, 28, 13, 13, 384, 6, 1, 1, 0.2, "iid"),
              (16, 23, 10, 10, 384, 6, 2, 2, 0.6, "structured")]


@pytest.mark.parametrize("h,w,hc,wc,C,H,B,B_max,keep,kind", SMALL_MAPS)
def test_every_selection_on_small_maps(h, w, hc, wc, C, H, B, B_max, keep, kind):
    test_every_selection_of_a_step_on_bit_identical_input(h, w, hc, wc, C, H, B, B_max, keep, kind, False, 0)


@pytest.mark.parametrize("resid_dtype", [0, 1])
@pytest.mark.parametrize("h,w,hc,wc,C,H,B,B_max,keep,kind", SMALL_MAPS)
def test_small_map_step_equals_the_separate_kernels(h, w, hc, wc, C, H, B, B_max, keep, kind, resid_dtype):
    """A free-running pruned step on a small map against the same step with its own kept sets forced, which runs the separate
    inverse-map, gather and restoration kernels: the arithmetic on every element is the same, so the maps are, bit for bit."""
    wl = I.Workload("small", L=2, C=C, H=H, B=B_max, sides=(hc, h), keep=(1.0, keep), cross_len=64, mlp_ratio=2, seed=812)
    mt = I.model_tensors(wl)
    k = O.kept_count(keep, h, w)
    ctx = fv.FvContext(wl.L, C, H, [(hc, wc), (h, w)], 0, B_max, k, mt, cross_len=64, mlp_ratio=2, device=DEV, resid_dtype=resid_dtype)
    for l in range(wl.L):
        for si in range(3):
            c = ctx.cache_view(l, si)
            c.copy_(_bf16_t(I.normal_bf16(820 + 3 * l + si, tuple(c.shape))))
    ctx.prepare_text(B)
    x = torch.from_numpy(I.token_map(830, B, h, w, C, kind)).to(DEV).to(ctx.x_dtype)
    trace = torch.full((wl.L, 3, B, k), -1, dtype=torch.int32, device=DEV)
    outs = []
    for forced in (None, None, trace):
        ctx.set_state(1, 0)
        outs.append(ctx.var_step(x, 1, keep, forced_idx=forced, idx_trace=trace if forced is None else None).clone())
    assert ctx.device_status() == 0
    assert torch.equal(outs[0], outs[1])
    assert torch.equal(outs[0], outs[2])
    ctx.close()


# How many restoration launches a step of 2 blocks x 2 sublayers makes: 1 with one launch between two sublayers (only the last one restores by itself);
# 7 where the last GEMM restores the kept rows (the other rows of every sublayer, and the sums of all but the last); 8 where a launch does.
@pytest.mark.parametrize("resid_dtype", [0, 1])
@pytest.mark.parametrize("h,w,C,H,B,keep,launches", [
    (16, 16, 1024, 16, 1, 0.6, 1), (16, 17, 1024, 16, 1, 0.6, 7), (16, 16, 1152, 18, 1, 0.6, 7), (16, 24, 384, 6, 1, 0.6, 1), (16, 25, 256, 4, 1, 0.6, 7), (16, 17, 512, 8, 1, 0.6, 7), (18, 18, 1920, 30, 2, 0.75, 7), (18, 18, 1920, 30, 2, 0.35, 1),
    (20, 28, 384, 6, 1, 0.9, 7), (20, 28, 384, 6, 1, 0.2, 1), (26, 31, 256, 2, 3, 0.16, 7), (26, 31, 256, 2, 3, 0.15, 8), (64, 64, 2048, 16, 1, 0.03, 8), (64, 64, 2048, 16, 1, 0.032, 7)])
def test_route_of_a_pruned_step(h, w, C, H, B, keep, launches, resid_dtype):
    wl = I.Workload("route", L=2, C=C, H=H, B=B, sides=(8, h), keep=(1.0, keep), mlp_ratio=1, seed=818)
    ctx = fv.FvContext(wl.L, C, H, [(8, 8), (h, w)], 0, B, O.kept_count(keep, h, w), I.model_tensors(wl), mlp_ratio=1, device=DEV, resid_dtype=resid_dtype)
    for l in range(wl.L):
        for si in range(2):
            ctx.cache_view(l, si).zero_()
    ctx.set_state(1, 0)
    fv.fv_profile_read()
    ctx.var_step(torch.zeros((B, h * w, C), dtype=ctx.x_dtype, device=DEV), 1, keep)
    assert fv.fv_profile_read()["restore"]["launches"] == launches and ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("resid_dtype", [0, 1])
@pytest.mark.parametrize("h,w,hc,wc,C,H,B,keep", [(26, 31, 10, 10, 256, 2, 3, 0.16), (48, 41, 13, 9, 1920, 30, 1, 0.33), (32, 32, 16, 16, 1024, 8, 3, 0.5),
                                                  (29, 29, 12, 12, 1152, 9, 2, 0.9985)])
def test_kept_rows_restored_by_the_last_gemm(h, w, hc, wc, C, H, B, keep, resid_dtype):
    """Kept rows added to the map by the GEMM that produces them: against the same step on one image at a time (tiles without an image
    boundary, other tile widths), as few kept rows as the route takes, a last tile of three rows, one token that is not kept.  Every selection behind the
    first takes its column sums from these GEMMs: with zero branches x never changes, so all of them must keep the first one's set."""
    wl = I.Workload("kept rows", L=2, C=C, H=H, B=B, sides=(hc, h), keep=(1.0, keep), cross_len=64, mlp_ratio=2, seed=815)
    k = O.kept_count(keep, h, w)
    assert k >= 128
    x = torch.from_numpy(I.token_map(831, B, h, w, C, "structured")).to(DEV)
    mt = I.model_tensors(wl)

    def ctx_of(tensors, images):
        ctx = fv.FvContext(wl.L, C, H, [(hc, wc), (h, w)], 0, images, k, tensors, cross_len=64, mlp_ratio=2, device=DEV, resid_dtype=resid_dtype)
        for l in range(wl.L):
            for si in range(3):
                c = ctx.cache_view(l, si)
                c.copy_(_bf16_t(I.normal_bf16(821 + 3 * l + si, (B,) + tuple(c.shape[1:])))[:images])
        ctx.prepare_text(images)
        ctx.set_state(1, 0)
        return ctx

    ctx = ctx_of(mt, B)
    x = x.to(ctx.x_dtype)
    trace = torch.full((wl.L, 3, B, k), -1, dtype=torch.int32, device=DEV)
    got = ctx.var_step(x, 1, keep, idx_trace=trace)
    ctx.set_state(1, 0)
    assert torch.equal(got, ctx.var_step(x, 1, keep, forced_idx=trace))        # the kept sets given: the same arithmetic
    assert ctx.device_status() == 0
    ctx.close()
    first_image = copy.copy(mt)
    first_image.mod, first_image.text = mt.mod[:, :1].copy(), mt.text[:1].copy()
    one = ctx_of(first_image, 1)
    alone = one.var_step(x[:1], 1, keep, forced_idx=trace[:, :, :1].contiguous())
    # other tiles: fp32 sums in another order, at most one bf16 rounding apart in any activation on the way
    err, cos = per_token_errors(got[:1].float().cpu().numpy(), alone.double().cpu().numpy())
    assert err <= MAX_ABS * (4 if resid_dtype else 1) and cos >= MIN_COS
    assert one.device_status() == 0
    one.close()
    zero = _zero_branch_tensors(wl)
    ctx = ctx_of(zero, B)
    for l in range(wl.L):
        for si in range(3):
            ctx.cache_view(l, si).zero_()
    assert torch.equal(ctx.var_step(x, 1, keep, idx_trace=trace), x)
    sets = trace.cpu().numpy()
    score = O.pts_score(x.double().cpu().numpy())
    tau = np.sort(score, axis=1)[:, ::-1][:, k - 1]
    first = O.pts_topk(score, k)
    for l in range(wl.L):
        for si in range(3):
            for b in range(B):
                diff = np.setxor1d(sets[l, si, b], first[b])
                assert np.all(np.abs(score[b, diff] - tau[b]) <= 1e-5 * tau[b])
    ctx.close()


@pytest.mark.parametrize("resid_dtype", [0, 1])
@pytest.mark.parametrize("sub", [0, 1])
@pytest.mark.parametrize("h,w,hc,wc,C,H,B,keep", [(26, 31, 10, 10, 256, 2, 3, 0.16), (48, 41, 13, 9, 1920, 30, 5, 0.3), (64, 64, 13, 9, 1024, 16, 2, 0.035)])
def test_kept_rows_restored_by_every_tile_of_the_last_gemm(h, w, hc, wc, C, H, B, keep, sub, resid_dtype):
    """Every tile that can restore the kept rows (one CTA of 64 ... 256 columns, that of 64 in both its builds, pairs of 128 and 256) against the oracle, with image boundaries inside
    its rows, a ragged last tile, and at the second shape more tiles than the GPU has SMs, so that accumulators and the tiles that turn rows are used again.
    One sublayer alone has a nonzero branch, so the map that the selections behind it see is the step's output: each must keep that map's set, for which it
    has only the column sums that the GEMM left.  The map is far from zero mean and its scores are dense: without one 32 x 32
    block of the sums the kept set of the first shape changes in 22 places, without that of the second in 14."""
    wl = I.Workload("every tile", L=2, C=C, H=H, B=B, sides=(hc, h), keep=(1.0, keep), mlp_ratio=1, seed=817)
    mt = _zero_branch_tensors(wl)
    if sub == 0:
        mt.w_o[0], mt.b_o[0] = I.normal_bf16(833, (C, C), 0.3), I.normal_bf16(834, (C,), 0.3)
    else:
        mt.w_fc2[0], mt.b_fc2[0] = I.normal_bf16(833, (C, C), 0.04), I.normal_bf16(834, (C,), 0.3)
    n, k = h * w, O.kept_count(keep, h, w)
    x = I.token_map(835, B, h, w, C, "iid") + np.float32(6.0)
    if resid_dtype:
        x = _bf16_round(x)
    ctx = fv.FvContext(wl.L, C, H, [(hc, wc), (h, w)], 0, B, k, mt, mlp_ratio=1, device=DEV, resid_dtype=resid_dtype)
    for l in range(wl.L):
        for si in range(2):
            ctx.cache_view(l, si).zero_()
    xd = torch.from_numpy(x).to(DEV).to(ctx.x_dtype)
    first = O.pts_topk(O.pts_score(x), k)
    forced = {(0, name): first for name in SUB_NAMES[2]}
    orc = O.VarOracle(1, C, H, [(hc, wc), (h, w)], cache_step=0, weights=helpers_oracle_weights(mt), B=B)
    orc.step = 1
    orc.cache[0] = {name: np.zeros((B, hc * wc, C)) for name in SUB_NAMES[2]}
    ref = orc.var_step(x, 1, keep, forced_idx=forced)
    kept = np.zeros((B, n), dtype=bool)
    np.put_along_axis(kept, first, True, axis=1)
    bound = MAX_ABS + (2.0 ** -8 * np.abs(ref).max() if resid_dtype else 0.0)            # (bf16 stream: one rounding)
    for path in (2, 3, 4, 5, 6, 7):
        trace = torch.full((wl.L, 2, B, k), -1, dtype=torch.int32, device=DEV)
        ctx.set_state(1, 0)
        assert fv.lib().fv_gemm_force_path(path) == 0
        try:
            got = ctx.var_step(xd, 1, keep, idx_trace=trace).double().cpu().numpy()
        finally:
            fv.lib().fv_gemm_force_path(0)
        assert ctx.device_status() == 0
        sets = trace.cpu().numpy()
        mine = np.zeros((B, n), dtype=bool)
        np.put_along_axis(mine, sets[0, sub].astype(np.int64), True, axis=1)
        assert np.array_equal(got[~mine], x[~mine].astype(np.float64)), path             # nothing but the kept rows is touched
        both = mine & kept
        assert both.sum() >= B * k - 4, path                                              # (the sets differ at near-ties alone: below)
        err, cos = per_token_errors(got[both], ref[both])
        assert err <= bound and cos >= MIN_COS, (path, err, cos)
        if not resid_dtype:
            assert per_token_errors(got[both] - x[both], ref[both] - x[both])[1] >= MIN_COS, path
        for l in range(wl.L):
            for si in range(2):
                score = O.pts_score(x if (l, si) <= (0, sub) else got)
                tau = np.sort(score, axis=1)[:, ::-1][:, k - 1]
                want = O.pts_topk(score, k)
                for b in range(B):
                    diff = np.setxor1d(sets[l, si, b], want[b])
                    assert np.all(np.abs(score[b, diff] - tau[b]) <= 1e-5 * tau[b]), (path, l, si, b, len(diff))
    ctx.close()


@pytest.mark.parametrize("resid_dtype", [0, 1])
def test_bytes_counted_for_the_gemms_and_the_restoration_of_a_step(resid_dtype):
    """fv_profile_read's dram_bytes of both classes is the sum over their launches of operands and results: for a residual GEMM the stream read
    and written (with the copy for the cache, or the column sums of the kept rows), for a pruned step's side stream the restoration
    of the other rows and the sum of its partials."""
    h, w, hc, wc, C, B, keep, L, ratio = 26, 31, 10, 10, 256, 3, 0.16, 2, 2
    wl = I.Workload("bytes", L=L, C=C, H=2, B=B, sides=(hc, h), keep=(1.0, keep), mlp_ratio=ratio, seed=816)
    n, nc, k, F, s = h * w, hc * wc, O.kept_count(keep, h, w), ratio * C, 4 if resid_dtype else 8
    ctx = fv.FvContext(L, C, 2, [(hc, wc), (h, w)], 0, B, nc + k, I.model_tensors(wl), mlp_ratio=ratio, device=DEV, resid_dtype=resid_dtype)
    xs = [torch.from_numpy(I.token_map(832, B, a, b, C, "structured")).to(DEV).to(ctx.x_dtype) for a, b in ((hc, wc), (h, w))]

    def gemms(M, out):          # QKV, out-projection and both MLP GEMMs of every block; out: bytes the two residual epilogues move, all blocks
        return L * 2 * (M * C + 3 * C * C + 3 * M * C + M * C + C * C + M * C + F * C + M * F + M * F + F * C) + out

    fv.fv_profile_read()
    ctx.var_step(xs[0], 0, 1.0)
    got = fv.fv_profile_read()
    assert got["gemm"]["dram_bytes"] == gemms(B * nc, 2 * L * (s + 2) * B * nc * C)
    assert got["restore"]["dram_bytes"] == 0
    ctx.var_step(xs[1], 1, keep)
    got = fv.fv_profile_read()
    blocks = sum((b * k + k - 1) // 128 - b * k // 128 + 1 for b in range(B))       # 128-row blocks of the compact rows, once per image they hold
    selections = 2 * L                                                               # the last one has no selection behind it
    assert got["gemm"]["dram_bytes"] == gemms(B * k, selections * s * B * k * C + (selections - 1) * 4 * C * blocks)
    assert got["restore"]["launches"] == 2 * selections - 1
    assert got["restore"]["dram_bytes"] == selections * B * C * (s * (n - k) + 2 * nc) + (selections - 1) * 4 * B * C * (-(-n // 32) + 1)
    assert ctx.device_status() == 0
    ctx.close()


def test_free_running_selection_matches_oracle_on_identical_input():
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i) for i in range(len(wl.sides))]
    orc, ref, tr = run_oracle(wl, mt, xs)
    ctx = make_ctx(wl, mt)
    got, traces = gpu_schedule(ctx, wl, xs, trace=True)
    first = wl.cache_step + 1
    names = SUB_NAMES[wl.n_sub]
    # block 0 / self-attention of every pruned step scores the step input itself: identical on both sides
    for i in range(first, len(xs)):
        idx_o = tr[i][(0, "attn")]["idx"]
        s_o = tr[i][(0, "attn")]["score"]
        idx_g = traces[i][0, 0].astype(np.int64)
        for b in range(wl.B):
            assert np.all(np.diff(idx_g[b]) > 0)                         # ascending, no duplicates
            diff = np.setxor1d(idx_g[b], idx_o[b])
            if len(diff):
                tau = np.sort(s_o[b])[::-1][idx_o.shape[1] - 1]
                assert np.all(np.abs(s_o[b, diff] - tau) <= 1e-5 * tau)
    # deeper sublayers see inputs that differ by bf16 rounding, so sets may differ near the threshold;
    # they must still be valid index sets and agree with the oracle on the bulk of the tokens
    agree = []
    for i in range(first, len(xs)):
        for l in range(wl.L):
            for si, name in enumerate(names):
                g, o = traces[i][l, si], tr[i][(l, name)]["idx"]
                for b in range(wl.B):
                    assert np.all(np.diff(g[b]) > 0) and g[b].min() >= 0 and g[b].max() < wl.tokens(i)
                    agree.append(len(np.intersect1d(g[b], o[b])) / o.shape[1])
    assert min(agree) >= 0.9
    # the pruned path is deterministic: same inputs, bit-identical outputs and kept sets, run to run
    # (column sums, K-split partial sums and the two-stream restoration all add in a fixed order)
    again, traces2 = gpu_schedule(ctx, wl, xs, trace=True)
    for i in range(len(xs)):
        assert np.array_equal(got[i], again[i])
        if traces[i] is not None:
            assert np.array_equal(traces[i], traces2[i])
    ctx.close()


def test_fused_selection_follows_the_separate_kernels_through_a_schedule():
    """The optional one-launch form of the in-step selection over a whole free-running schedule (two pruned steps,
    two blocks): given the same kept sets it must give the token maps of the separate kernels bit for bit (their
    arithmetic on x is identical; only the column sums are added in another order), and twice in a row the same bits."""
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i, "structured") for i in range(len(wl.sides))]
    ctx = make_ctx(wl, mt)
    ref, tr_ref = gpu_schedule(ctx, wl, xs, trace=True)
    assert fv.lib().fv_step_fused_selection(1) == 0
    try:
        got, tr = gpu_schedule(ctx, wl, xs, trace=True)
        again, tr2 = gpu_schedule(ctx, wl, xs, trace=True)
    finally:
        fv.lib().fv_step_fused_selection(0)
    same_sets = True
    for i in range(len(xs)):
        assert np.array_equal(got[i], again[i])
        if tr[i] is not None:
            assert np.array_equal(tr[i], tr2[i])
            g, r = tr[i].astype(np.int64), tr_ref[i].astype(np.int64)
            assert np.all(np.diff(g, axis=-1) > 0) and g.min() >= 0 and g.max() < wl.tokens(i)
            same_sets = same_sets and np.array_equal(g, r)
        if same_sets:
            assert np.array_equal(got[i], ref[i]), i
        else:
            err, cos = per_token_errors(got[i], ref[i])
            assert err <= MAX_ABS and cos >= MIN_COS
    ctx.close()


# ------------------------------------------------------------------ bf16 residual stream (fv_config.resid_dtype = 1)
def _bf16_round(a):
    return I.bf16_bits_to_f32(I.to_bf16_bits(a))


def test_bf16_residual_stream_schedule_against_the_oracle():
    """The token maps of fv_var_step in bf16: every kernel that touches the stream (column sums, scores, gather,
    restoration, the residual epilogue of the unpruned steps) reads and writes bf16 and computes in fp32.  Inputs are
    bf16-representable on both sides; the oracle stays fp64.  Each of the U updates of a step rounds the stream once
    (<= 2^-9 relative), so the bound is the usual 3e-2 of the branch arithmetic plus U * 2^-9 * max|x|; the first
    selection of every pruned step sees identical input and must keep the oracle's set."""
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [_bf16_round(I.step_input(wl, i, "structured")) for i in range(len(wl.sides))]
    orc, ref, tr = run_oracle(wl, mt, xs)
    forced = [trace_to_index_tensor(wl, tr[i]) if wl.keep[i] < 1.0 else None for i in range(len(xs))]
    ctx = make_ctx(wl, mt, resid_dtype=1)
    updates = wl.L * wl.n_sub
    worst = 0.0
    for mode in ("forced", "free"):
        ctx.reset()
        for i, x in enumerate(xs):
            xd = torch.from_numpy(x).to(DEV).to(torch.bfloat16)
            f = t = None
            if wl.keep[i] < 1.0:
                if mode == "forced":
                    f = torch.from_numpy(forced[i]).to(DEV)
                else:
                    t = torch.zeros((wl.L, wl.n_sub, wl.B, forced[i].shape[-1]), dtype=torch.int32, device=DEV)
            got = ctx.var_step(xd, i, wl.keep[i], forced_idx=f, idx_trace=t)
            assert got.dtype == torch.bfloat16
            got = got.float().cpu().numpy()
            if mode == "forced":
                err, cos = per_token_errors(got, ref[i])
                bound = MAX_ABS + updates * 2.0 ** -9 * np.abs(ref[i]).max()
                worst = max(worst, err)
                assert err <= bound and cos >= MIN_COS, (i, err, bound, cos)
            elif t is not None:
                idx_g = t[0, 0].cpu().numpy().astype(np.int64)
                idx_o, s_o = tr[i][(0, "attn")]["idx"], tr[i][(0, "attn")]["score"]
                for b in range(wl.B):
                    diff = np.setxor1d(idx_g[b], idx_o[b])
                    tau = np.sort(s_o[b])[::-1][idx_o.shape[1] - 1]
                    assert np.all(np.abs(s_o[b, diff] - tau) <= 1e-5 * tau)
        assert ctx.device_status() == 0 and ctx.state() == (len(xs), orc.kv_len)
    print(f"bf16 residual stream, tiny schedule: worst max-abs error {worst:.4g}")
    # what the bf16 stream does not take
    with pytest.raises(fv.FvError) as e:
        fv.FvContext(wl.L, wl.C, wl.H, [(s, s) for s in wl.sides], wl.cache_step, wl.B, 64, mt, device=DEV, granularity=1, resid_dtype=1)
    assert e.value.code == 4
    ctx.close()


@pytest.mark.parametrize("h,w,hc,wc,C,H,B,B_max,keep", [(64, 64, 32, 32, 2048, 16, 2, 2, 0.2), (33, 31, 10, 10, 256, 4, 3, 4, 0.5),
                                                      (128, 128, 48, 48, 2048, 16, 1, 1, 0.2), (33, 31, 10, 10, 256, 4, 3, 4, 0.12),
                                                      (64, 64, 32, 32, 2048, 16, 2, 2, 0.03), (128, 128, 48, 48, 2048, 16, 1, 1, 0.0077)])
def test_bf16_residual_stream_every_selection_on_bit_identical_input(h, w, hc, wc, C, H, B, B_max, keep):
    """The zero-branch step (see test_every_selection_of_a_step_on_bit_identical_input) with a bf16 stream: x + 0 is
    exact in bf16 too, so every one of the six selections -- five of them from the column sums the bf16 restoration
    left -- must keep the oracle's set of the (bf16-representable) map."""
    wl = I.Workload("zero-branch", L=2, C=C, H=H, B=B_max, sides=(hc, h), keep=(1.0, keep), cross_len=64, mlp_ratio=1, seed=811)
    mt = _zero_branch_tensors(wl)
    n, k = h * w, O.kept_count(keep, h, w)
    x = _bf16_round(I.token_map(900 + h, B, h, w, C, "structured"))
    ctx = fv.FvContext(wl.L, C, H, [(hc, wc), (h, w)], 0, B_max, k, mt, cross_len=64, mlp_ratio=1, device=DEV, resid_dtype=1)
    for l in range(wl.L):
        for si in range(3):
            ctx.cache_view(l, si).zero_()
    ctx.set_state(1, 0)
    ctx.prepare_text(B)
    trace = torch.full((wl.L, 3, B, k), -1, dtype=torch.int32, device=DEV)
    got = ctx.var_step(torch.from_numpy(x).to(DEV).to(torch.bfloat16), 1, keep, idx_trace=trace).float().cpu().numpy()
    assert ctx.device_status() == 0
    assert np.array_equal(got, x)
    score_o = O.pts_score(x)
    idx_o = O.pts_topk(score_o, k)
    tau = np.sort(score_o, axis=1)[:, ::-1][:, k - 1]
    idx_g = trace.cpu().numpy().astype(np.int64)
    for l in range(wl.L):
        for si in range(3):
            for b in range(B):
                g = idx_g[l, si, b]
                assert np.all(np.diff(g) > 0) and g[0] >= 0 and g[-1] < n
                diff = np.setxor1d(g, idx_o[b])
                assert np.all(np.abs(score_o[b, diff] - tau[b]) <= 1e-5 * tau[b]), (l, si, b)
    ctx.close()


# ------------------------------------------------------------------ per-step granularity (the coarser variant)
def check_step_granularity(wl, kind="iid"):
    """One selection and one restoration around the whole stack of blocks, against the oracle's variant of
    the same name: forced indices for the floating point, free running for the indices (the selection
    sees the step input itself, identical on both sides)."""
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i, kind) for i in range(len(wl.sides))]
    orc = O.VarOracle(wl.L, wl.C, wl.H, [(s, s) for s in wl.sides], cache_step=wl.cache_step,
                      weights=helpers_oracle_weights(mt), B=wl.B, cross_len=wl.cross_len, granularity="step")
    ref, tr = [], []
    for i, x in enumerate(xs):
        t = {}
        ref.append(orc.var_step(x, i, wl.keep[i], trace=t))
        tr.append(t)
    ctx = make_ctx(wl, mt, granularity=1)
    for mode in ("forced", "free"):
        ctx.reset()
        for i, x in enumerate(xs):
            xd = torch.from_numpy(x).to(DEV)
            f = t = None
            if wl.keep[i] < 1.0:
                idx_o = tr[i][("step",)]["idx"]
                if mode == "forced":
                    f = torch.from_numpy(idx_o.astype(np.int32)).to(DEV)
                else:
                    t = torch.zeros(idx_o.shape, dtype=torch.int32, device=DEV)
            got = ctx.var_step(xd, i, wl.keep[i], forced_idx=f, idx_trace=t).cpu().numpy()
            if t is not None:
                idx_g = t.cpu().numpy().astype(np.int64)
                s_o = tr[i][("step",)]["score"]
                same = True
                for b in range(wl.B):
                    assert np.all(np.diff(idx_g[b]) > 0)
                    diff = np.setxor1d(idx_g[b], idx_o[b])
                    if len(diff):
                        same = False
                        tau = np.sort(s_o[b])[::-1][idx_o.shape[1] - 1]
                        assert np.all(np.abs(s_o[b, diff] - tau) <= 1e-5 * tau), "index mismatch away from a near-tie"
                if not same:
                    continue        # a near-tie went the other way: the floating-point check ran in forced mode
            err, cos = per_token_errors(got, ref[i])
            assert err <= MAX_ABS and cos >= MIN_COS, f"{mode} step {i} side {wl.sides[i]}: max-abs {err:.4g}, cos {cos:.6f}"
            if wl.keep[i] < 1.0:     # rows that were not kept are exact copies of the cached output map
                hc = wl.sides[wl.cache_step]
                src = O.nearest_source(wl.sides[i], wl.sides[i], hc, hc)
                cache = ctx.cache_view(0, 0, wl.B).cpu().numpy()
                idx_used = tr[i][("step",)]["idx"] if mode == "forced" else idx_g
                for b in range(wl.B):
                    rest = np.setdiff1d(np.arange(wl.tokens(i)), idx_used[b])
                    assert np.array_equal(got[b, rest], cache[b, src[rest]])
        assert ctx.device_status() == 0 and ctx.state() == (len(xs), orc.kv_len)
    ctx.close()


def test_step_granularity_tiny_schedule():
    check_step_granularity(I.WORKLOADS["tiny"])
    check_step_granularity(I.WORKLOADS["tiny"], kind="structured")


def test_step_granularity_infinity_shape_with_cross_attention():
    base = I.WORKLOADS["infinity_2b_1k"]
    sides = (1, 2, 4, 8, 12, 16, 24)
    wl = I.Workload("inf-short", L=2, C=base.C, H=base.H, B=2, sides=sides,
                    keep=(1.0, 1.0, 1.0, 1.0, 1.0, 0.6, 0.4), cross_len=64, seed=base.seed)
    check_step_granularity(wl)


@pytest.mark.parametrize("granularity", [0, 1])
def test_skipped_step_keep_ratio_zero(granularity):
    """keep_ratio = 0 (the paper's 100 % pruning ratio): the output is an exact copy of rows of the caching
    step's output map (nearest interpolation), the KV cache does not grow, the next pruned step still runs."""
    base = I.WORKLOADS["tiny"]
    keep = tuple(base.keep[:8]) + (0.0, 0.5)                  # sides ..., 10 (cache step 7), 13 skipped, 16 pruned
    wl = I.Workload("tiny-skip", L=base.L, C=base.C, H=base.H, B=base.B, sides=base.sides, keep=keep, seed=base.seed)
    assert wl.cache_step == 7
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i) for i in range(len(wl.sides))]
    orc = O.VarOracle(wl.L, wl.C, wl.H, [(s, s) for s in wl.sides], cache_step=wl.cache_step, weights=helpers_oracle_weights(mt),
                      B=wl.B, cross_len=wl.cross_len, granularity="step" if granularity else "sublayer")
    ctx = make_ctx(wl, mt, granularity=granularity)
    outs = []
    for i, x in enumerate(xs):
        tr = {}
        ref = orc.var_step(x, i, wl.keep[i], trace=tr)
        forced = None
        if 0.0 < wl.keep[i] < 1.0:
            forced = torch.from_numpy(tr[("step",)]["idx"].astype(np.int32) if granularity else trace_to_index_tensor(wl, tr)).to(DEV)
        got = ctx.var_step(torch.from_numpy(x).to(DEV), i, wl.keep[i], forced_idx=forced).cpu().numpy()
        outs.append(got)
        err, cos = per_token_errors(got, ref)
        assert err <= MAX_ABS and cos >= MIN_COS, (i, err, cos)
        assert ctx.state() == (i + 1, orc.kv_len)
    src = O.nearest_source(13, 13, 10, 10)
    assert np.array_equal(outs[8], outs[7][:, src])          # a copy of the cached map's rows, bit for bit
    assert ctx.device_status() == 0
    ctx.close()


def test_non_square_maps_and_partial_batch():
    """Token maps need not be square, and a call may use fewer images than the context was built for."""
    hw = [(1, 1), (2, 3), (3, 5), (5, 8), (7, 12), (10, 17)]
    keep = [1.0, 1.0, 1.0, 1.0, 0.5, 0.3]
    L, C, H, B_max, B = 2, 128, 2, 3, 2
    wl = I.Workload("rect", L=L, C=C, H=H, B=B_max, sides=tuple(h for h, _ in hw), keep=tuple(keep), cross_len=8, seed=77)
    mt = I.model_tensors(wl)
    w = helpers_oracle_weights(mt)
    w = dict(w); w["mod"] = w["mod"][:, :B]; w["text"] = w["text"][:B]
    orc = O.VarOracle(L, C, H, hw, cache_step=3, weights=w, B=B, cross_len=8)
    cap = sum(O.kept_count(r, h, ww) if r < 1 else h * ww for r, (h, ww) in zip(keep, hw))
    ctx = fv.FvContext(L, C, H, hw, 3, B_max, cap, mt, cross_len=8, device=DEV)
    for i, (h, ww) in enumerate(hw):
        x = I.token_map(500 + i, B, h, ww, C)
        tr = {}
        ref = orc.var_step(x, i, keep[i], trace=tr)
        forced = None
        if keep[i] < 1.0:
            forced = torch.from_numpy(np.stack([np.stack([tr[(l, s)]["idx"] for s in SUB_NAMES[3]]) for l in range(L)]).astype(np.int32)).to(DEV)
        got = ctx.var_step(torch.from_numpy(x).to(DEV), i, keep[i], forced_idx=forced).cpu().numpy()
        err, cos = per_token_errors(got, ref)
        assert err <= MAX_ABS and cos >= MIN_COS, (i, err, cos)
    assert ctx.device_status() == 0 and ctx.state() == (len(hw), orc.kv_len)
    ctx.close()


def test_keep_ratio_one_is_the_unpruned_path_and_is_deterministic():
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i) for i in range(len(wl.sides))]
    wl_full = I.Workload("tiny-full", L=wl.L, C=wl.C, H=wl.H, B=wl.B, sides=wl.sides, keep=(1.0,) * len(wl.sides), seed=wl.seed)
    _, ref, _ = run_oracle(wl_full, mt, xs)
    ctx = make_ctx(wl, mt, unpruned=True)
    a, _ = gpu_schedule(ctx, wl_full, xs)
    b, _ = gpu_schedule(ctx, wl_full, xs)
    for i in range(len(xs)):
        assert np.array_equal(a[i], b[i])                                # bit-identical run to run
        err, cos = per_token_errors(a[i], ref[i])
        assert err <= MAX_ABS and cos >= MIN_COS
    ctx.close()


def test_state_and_argument_errors():
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    ctx = make_ctx(wl, mt)
    x0 = torch.from_numpy(I.step_input(wl, 0)).to(DEV)
    x1 = torch.from_numpy(I.step_input(wl, 1)).to(DEV)
    with pytest.raises(fv.FvError) as e:
        ctx.var_step(x1, 1, 1.0)                                         # out of order
    assert e.value.code == 2
    with pytest.raises(fv.FvError) as e:
        ctx.var_step(x0, 0, 0.5)                                         # pruned before the cache step
    assert e.value.code == 2
    with pytest.raises(fv.FvError) as e:
        ctx.var_step(x0, 0, 0.0)                                         # nothing cached yet to interpolate
    assert e.value.code == 2
    with pytest.raises(fv.FvError) as e:
        ctx.var_step(x0, 0, -0.1)
    assert e.value.code == 1
    ctx.var_step(x0, 0, 1.0)
    assert ctx.state() == (1, 1)
    ctx.set_state(9, ctx.kv_capacity)                                    # cache full: the next step cannot fit
    x9 = torch.from_numpy(I.step_input(wl, 9)).to(DEV)
    with pytest.raises(fv.FvError) as e:
        ctx.var_step(x9, 9, 0.5)
    assert e.value.code == 3
    ctx.close()


def test_an_expired_device_wait_is_reported_not_fatal():
    """The library's kernels never wait without a limit: a wait that nothing ends gives up after its limit, leaves a
    code in the context's status word and the kernel returns normally.  The self-test kernel waits 50 microseconds
    on a barrier nobody completes; fv_device_status must report FV_ERR_TIMEOUT with its code, clear the word, and
    the context must go on working (a full schedule afterwards still matches the run before it)."""
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i) for i in range(len(wl.sides))]
    ctx = make_ctx(wl, mt)
    before, _ = gpu_schedule(ctx, wl, xs)
    ctx.selftest_expired_wait(50_000)
    assert ctx.device_status_pair() == (6, 105)          # FV_ERR_TIMEOUT, the self-test's code
    assert ctx.device_status_pair() == (0, 0)            # cleared by the read
    with pytest.raises(fv.FvError) as e:
        ctx.selftest_expired_wait(0)                     # a limit is mandatory
    assert e.value.code == 1
    after, _ = gpu_schedule(ctx, wl, xs)
    for a, b in zip(before, after):
        assert np.array_equal(a, b)
    ctx.close()


def test_an_index_outside_the_map_is_clamped_and_reported():
    """A kept-row index outside [0, n) (a caller's mistake in forced-index mode) must not become a read outside the
    token map: the gather clamps it into the map and leaves code 41 in the status word."""
    B, n, C, k = 2, 50, 256, 4
    x = I.normal(321, (B, n, C))
    idx = np.array([[0, 7, 49, 50], [-3, 2, 10, 4999]], dtype=np.int32)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = fv.fv_gather_ln(torch.from_numpy(x).to(DEV), torch.from_numpy(idx).to(DEV), None, None, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 41
    clamped = np.clip(idx, 0, n - 1).astype(np.int64)
    ref = O.layernorm(O.pts_gather(x.astype(np.float64), clamped))
    err, cos = per_token_errors(got.float().cpu().numpy(), ref)
    assert err <= MAX_ABS and cos >= MIN_COS
    status.zero_()
    fv.fv_gather_ln(torch.from_numpy(x).to(DEV), torch.from_numpy(clamped.astype(np.int32)).to(DEV), None, None, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0


def test_step_with_host_buffers_equals_the_device_call():
    """fv_var_step_host (pinned host token maps in, host result out) gives the bits of fv_var_step."""
    wl = I.WORKLOADS["tiny"]
    mt = I.model_tensors(wl)
    xs = [I.step_input(wl, i) for i in range(len(wl.sides))]
    ctx = make_ctx(wl, mt)
    ref, _ = gpu_schedule(ctx, wl, xs)
    ctx.reset()
    hins = [torch.from_numpy(x).pin_memory() for x in xs]
    houts = [torch.empty_like(h).pin_memory() for h in hins]
    for rep in range(2):          # all steps enqueued back to back: copies and steps overlap across calls
        ctx.reset()
        for h in houts:
            h.zero_()
        for i in range(len(xs)):
            ctx.var_step_host(hins[i], i, wl.keep[i], houts[i])
        ctx.host_io_flush()
        torch.cuda.synchronize()
        for i in range(len(xs)):
            assert np.array_equal(houts[i].numpy(), ref[i]), (rep, i)
    hin, hout = hins[0], houts[0]
    assert ctx.device_status() == 0
    with pytest.raises(fv.FvError) as e:      # staging too small
        fv._check(fv.lib().fv_var_step_host(ctx.ctx, hin.data_ptr(), 1, 0, 1.0, hout.data_ptr(), 1024, 16, None), "fv_var_step_host")
    assert e.value.code == 3
    ctx.close()
