"""The work whose speed is tracked: whole scale schedules through FvContext, the paper's two stand-alone calls
(prune_select, restore) and the stages of the generation loop around a scale step.

A case is a dict of plain values; `listed()` names the standing ones, `draw(rng)` gives more of the same ranges.
Shapes are those of `paper_2503_23367_b200.inputs.WORKLOADS` unless a comment says otherwise.
"""
from __future__ import annotations

import math

import torch

from paper_2503_23367_b200 import binding as fv
from paper_2503_23367_b200 import inputs as I

L2_BYTES = 126e6                 # weights that fit here need not be read again at every scale step


# ------------------------------------------------------------------------------------------------ the cases
def _text(values) -> str:
    return ",".join(f"{v:g}" for v in values)


def _schedule(name, L, C, H, B, h, w, keep, text=0, stream="fp32", rotary=False, interp=0, host=False):
    """One pass = every scale step of one batch, in order.  `keep` are the ratios of the last len(keep) steps (1 before
    them).  stream: type of the token maps; rotary: cosine attention + rotary positions; interp: 0 nearest,
    1 bilinear, 2 bicubic; host: token maps in pinned host memory."""
    c = {"kind": "schedule", "L": L, "C": C, "H": H, "B": B, "h": _text(h), "w": _text(w), "keep": _text(keep), "text": text,
         "stream": stream, "rotary": bool(rotary), "interp": interp, "host": bool(host)}
    return dict(c, name=name) if name else c


def _workload(name, workload, B=None, **options):
    wl = I.WORKLOADS[workload]
    return _schedule(name, wl.L, wl.C, wl.H, B or wl.B, wl.sides, wl.sides, [k for k in wl.keep if k < 1.0], text=wl.cross_len, **options)


def _select(name, B, h, w, C, keep):
    c = {"kind": "select", "B": B, "h": h, "w": w, "C": C, "keep": keep}
    return dict(c, name=name) if name else c


def _restore(name, B, h, w, hc, wc, C, keep, interp=0):
    c = {"kind": "restore", "B": B, "h": h, "w": w, "hc": hc, "wc": wc, "C": C, "keep": keep, "interp": interp}
    return dict(c, name=name) if name else c


def _stages(name, B, h, w, h2, w2, C, V, d):
    c = {"kind": "stages", "B": B, "h": h, "w": w, "h2": h2, "w2": w2, "C": C, "V": V, "d": d}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model: every call is a handful of rows, so launches and latency are all there is
        _workload("tiny", "tiny"),
        # class-conditional 256-pixel images: one image for an interactive user, and a batch
        _workload("d16_256px_one", "var_d16_256", B=1),
        _workload("d16_256px", "var_d16_256"),
        # 512-pixel images from a serving process whose token maps come from and go to pinned host memory
        _workload("d30_512px_host", "var_d30_512", host=True),
        # text-to-image at 1024 pixels: the ordinary case
        _workload("infinity_1k", "infinity_2b_1k"),
        # the paper's own ratios for it (two skipped steps), the cache interpolated bilinearly
        _workload("infinity_1k_paper_bilinear", "infinity_2b_1k_paper", interp=1),
        # token maps in bf16, cosine attention and rotary positions: what the pruned backbone itself computes
        _workload("infinity_1k_bf16_rotary", "infinity_2b_1k", stream="bf16", rotary=True),
        # zero-shot 2K: the largest
        _workload("infinity_2k", "infinity_2b_2k"),
        # selection alone for a caller with its own transformer: the largest map, and a small ragged batch
        _select("select_128x128", 1, 128, 128, 2048, 0.2),
        _select("select_small_ragged", 3, 13, 18, 1920, 0.6),
        # restoration alone: 64x64 map of the 1024-pixel schedule from its caching step
        _restore("restore_64x64", 2, 64, 64, 32, 32, 2048, 0.2),
        # between two steps of the generation loop: head, greedy tokens, residual accumulation, next token map
        _stages("stages_48_to_64", 2, 48, 48, 64, 64, 2048, 4096, 32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_schedule(rng):
    C, H = rng.choice([(256, 4), (512, 8), (1024, 16), (1024, 8), (1536, 12), (1920, 30), (2048, 16)])
    text = rng.choice([0, 0, 8 * _log(rng, 4, 64)])
    steps = rng.randint(6, 14)
    last = _log(rng, 8, 100)
    aspect = rng.choice([1.0, 1.0, 0.75, 1.5])
    h, w = [1], [1]
    for i in range(1, steps):
        side = last ** (i / (steps - 1))
        a, b = max(1, int(round(side))), max(1, int(round(side * aspect)))
        if (a, b) != (h[-1], w[-1]):
            h.append(max(a, h[-1]))
            w.append(max(b, w[-1]))
    pruned = rng.randint(1, min(4, len(h) - 2))
    keep = sorted((round(rng.uniform(0.15, 0.8), 2) for _ in range(pruned)), reverse=True)
    bf16 = rng.random() < 0.25
    case = _schedule(None, _log(rng, 2, 32), C, H, rng.choice([1, 1, 2, 3, 4, 8]), h, w, keep, text=text, stream="bf16" if bf16 else "fp32",
                     rotary=rng.random() < 0.25, interp=0 if bf16 else rng.choice([0, 0, 0, 1, 2]), host=rng.random() < 0.15)
    top = work(_workload("", "infinity_2b_2k"))
    while case["L"] > 1 or case["B"] > 1:
        mine = work(case)
        if mine["flops"] <= 0.7 * top["flops"] and mine["bytes"] <= 0.7 * top["bytes"]:
            break
        case["L"], case["B"] = (max(1, case["L"] // 2), case["B"]) if case["L"] > 1 else (case["L"], case["B"] // 2)
    return case


def draw(rng):
    kind = rng.choice(["schedule"] * 5 + ["select", "select", "restore", "stages"])
    if kind == "schedule":
        return _draw_schedule(rng)
    C = rng.choice([256, 768, 1024, 1920, 2048])
    B = rng.choice([1, 1, 2, 3, 4, 8])
    h = _log(rng, 8, 128 if B <= 2 else 64)
    w = max(4, min(128, int(round(h * rng.choice([1.0, 1.0, 0.7, 1.4])))))
    keep = round(rng.uniform(0.1, 0.9), 3)
    if kind == "select":
        return _select(None, B, h, w, C, keep)
    if kind == "restore":
        return _restore(None, B, h, w, max(1, h * rng.randint(3, 8) // 10), max(1, w * rng.randint(3, 8) // 10), C, keep, rng.choice([0, 0, 0, 1, 2]))
    grow = rng.uniform(1.1, 1.6)
    h, w = min(h, 64), min(w, 64)
    return _stages(None, B, h, w, min(128, int(h * grow) + 1), min(128, int(w * grow) + 1), C, rng.choice([1024, 4096]), rng.choice([16, 32]))


# ------------------------------------------------------------------------------------------------ what a case is
def _sizes(case):
    h, w = [int(v) for v in case["h"].split(",")], [int(v) for v in case["w"].split(",")]
    tail = [float(v) for v in case["keep"].split(",")]
    keep = [1.0] * (len(h) - len(tail)) + tail
    kept = [0 if r == 0.0 else min(a * b, max(1, math.ceil(r * a * b - 1e-9))) for a, b, r in zip(h, w, keep)]
    return h, w, keep, kept


def work(case):
    B, C = case["B"], case["C"]
    if case["kind"] == "select":
        n = case["h"] * case["w"]
        return {"bytes": 4.0 * B * n * C + 4.0 * B * (2 * n + case["keep"] * n), "flops": 4.0 * B * n * C}
    if case["kind"] == "restore":
        n, nc = case["h"] * case["w"], case["hc"] * case["wc"]
        k = math.ceil(case["keep"] * n)
        return {"bytes": 2.0 * B * C * (n + k + nc) + 4.0 * B * k, "flops": 0.0}
    if case["kind"] == "stages":
        n, n2, V, d = case["h"] * case["w"], case["h2"] * case["w2"], case["V"], case["d"]
        return {"bytes": 4.0 * B * n * C + 2.0 * V * C + 4.0 * B * n * V + 4.0 * B * n * (1 + d) + 4.0 * V * d + 4.0 * n2 * C + 4.0 * B * n2 * C,
                "flops": 2.0 * B * n * C * V + 2.0 * B * n2 * d * C}
    # a schedule: per step the map in and out once, the weights once (they do not stay on the chip from one step to the
    # next unless the whole model fits the L2 cache), the keys and values of the earlier steps and of the text once, and at a
    # pruned step the sublayer caches once
    h, w, keep, kept = _sizes(case)
    L, text = case["L"], case["text"]
    weights = 2.0 * L * C * C * (12 + (2 if text else 0))
    elem = 2 if case["stream"] == "bf16" else 4
    nc = max([a * b for a, b, r in zip(h, w, keep) if r == 1.0])
    byt, flops, kv, first = 0.0, 0.0, 0, True
    for a, b, r, k in zip(h, w, keep, kept):
        byt += elem * B * a * b * C * (2 if k else 1)
        if not k:
            byt += 4.0 * B * nc * C
            continue
        if first or weights > L2_BYTES:
            byt += weights
        first = False
        flops += 24.0 * L * B * k * C * C + 4.0 * L * B * k * (kv + k) * C
        byt += 4.0 * L * B * C * (kv + k)
        if text:
            flops += 4.0 * L * B * k * C * C + 4.0 * L * B * k * text * C
            byt += 4.0 * L * B * text * C
        if r < 1.0:
            byt += 2.0 * L * (3 if text else 2) * B * nc * C
        kv += k
    if text:                                     # keys and values of the text, once per schedule
        flops += 8.0 * C * C * L * B * text / 2
        byt += 4.0 * L * C * C + 2.0 * B * text * C
    return {"bytes": byt, "flops": flops}


def tolerance(case):
    if case["kind"] == "select":                 # fp32 sums in another order; a kept token may change at a near-tie
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    if case["kind"] == "restore":                # rows are copied (exact) or interpolated in fp32 and rounded to bf16
        return "exact" if case["interp"] == 0 else {"rel": 4e-3, "max": 2e-2}
    if case["kind"] == "stages":                 # bf16 GEMM; a token (one codebook row) may change where two logits tie
        return {"rel": 0.03, "max": 0.99, "differ": 1e-3}
    # A schedule through other GEMM tiles (its fp32 sums in another order, so other bf16 roundings) moved its maps by at most
    # rel 3.5e-3, max 5e-2 over the listed and a dozen drawn cases with an fp32 stream, and rel 1.2e-2, max 8e-2 with a bf16 stream.
    return {"rel": 0.03, "max": 0.3} if case["stream"] == "bf16" else {"rel": 1e-2, "max": 0.2}


# ------------------------------------------------------------------------------------------------ inputs
class _Tensors:
    """Random weights of the model's shapes (bf16 N(0, 0.02^2)), as `FvContext` takes them; gates and modulation N(0, 0.1^2), so
    that a branch adds to the residual stream what one adds in a trained model, a fraction of the stream."""

    def __init__(self, case, g):
        L, B, C = case["L"], case["B"], case["C"]
        F, text = 4 * C, case["text"]

        def r(*shape, std=0.02):
            return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)

        self.w_qkv, self.b_qkv = [r(3 * C, C) for _ in range(L)], [r(3 * C) for _ in range(L)]
        self.w_o, self.b_o = [r(C, C) for _ in range(L)], [r(C) for _ in range(L)]
        self.w_fc1, self.b_fc1 = [r(F, C) for _ in range(L)], [r(F) for _ in range(L)]
        self.w_fc2, self.b_fc2 = [r(C, F) for _ in range(L)], [r(C) for _ in range(L)]
        self.w_q_x = [r(C, C) for _ in range(L)] if text else []
        self.w_kv_x = [r(2 * C, C) for _ in range(L)] if text else []
        self.w_o_x = [r(C, C) for _ in range(L)] if text else []
        self.mod = torch.randn(L, B, 6, C, generator=g, device="cuda").mul_(0.1)
        self.text = r(B, text, C, std=1.0) if text else None


def _token_map(g, B, h, w, C, textured):
    """A map with flat and textured regions: a smooth field, a little noise everywhere and strong noise on `textured` tokens of
    every image.  A pruned step keeps as many tokens as there are textured ones: the ratio fits the image, and its scores
    leave a gap at the threshold, so that rounding alone does not change which tokens a free-running schedule keeps."""
    coarse = torch.randn(B, C, -(-h // 8), -(-w // 8), generator=g, device="cuda")
    smooth = torch.nn.functional.interpolate(coarse, size=(h, w), mode="bilinear").permute(0, 2, 3, 1).reshape(B, h * w, C)
    edge = torch.rand(B, h * w, generator=g, device="cuda").argsort(dim=1).unsqueeze(2) < textured
    return smooth.add(torch.randn(B, h * w, C, generator=g, device="cuda") * (0.1 + 1.4 * edge)).contiguous()


def _prepare_schedule(case, g):
    h, w, keep, kept = _sizes(case)
    B, C = case["B"], case["C"]
    cache_step = sum(r == 1.0 for r in keep) - 1
    scale = torch.rand(case["L"], case["H"], generator=g, device="cuda").mul_(8).add_(4) if case["rotary"] else None
    bf16 = case["stream"] == "bf16"
    ctx = fv.FvContext(case["L"], C, case["H"], list(zip(h, w)), cache_step, B, sum(kept), _Tensors(case, g), cross_len=case["text"],
                       rope_base=10000.0 if case["rotary"] else 0.0, qk_scale=scale, interp_mode=case["interp"], resid_dtype=1 if bf16 else 0)
    maps = [_token_map(g, B, a, b, C, k if 0 < k < a * b else a * b // 5).to(torch.bfloat16 if bf16 else torch.float32) for a, b, k in zip(h, w, kept)]
    if case["host"]:
        maps = [m.cpu().pin_memory() for m in maps]
        outs = [torch.empty_like(m).pin_memory() for m in maps]
    else:
        outs = [torch.empty_like(m) for m in maps]
    return {"kind": "schedule", "ctx": ctx, "maps": maps, "outs": outs, "keep": keep, "host": case["host"]}


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "schedule":
        return _prepare_schedule(case, g)
    B, C, h, w = case["B"], case["C"], case["h"], case["w"]
    if case["kind"] == "select":
        return dict(case, x=_token_map(g, B, h, w, C, h * w // 5), ws=fv.fv_prune_select_workspace(B, h * w, C, "cuda"))
    if case["kind"] == "restore":
        k = fv.fv_k_for(case["keep"], h, w)
        idx = torch.rand(B, h * w, generator=g, device="cuda").topk(k, dim=1).indices.sort(dim=1).values.int().contiguous()

        def r(n):
            return torch.randn(B, n, C, generator=g, device="cuda").bfloat16()

        return dict(case, cache=r(case["hc"] * case["wc"]), pivots=r(k), idx=idx, out=torch.empty(B, h * w, C, dtype=torch.bfloat16, device="cuda"))
    V, d = case["V"], case["d"]

    def n(*shape, std=1.0):
        return torch.randn(*shape, generator=g, device="cuda").mul_(std)

    hp, wp = max(1, h * 3 // 4), max(1, w * 3 // 4)
    return dict(case, y=_token_map(g, B, h, w, C, h * w // 5), mod_head=n(B, 2, C, std=0.3), w_head=n(V, C, std=0.08).bfloat16(), b_head=n(V, std=0.02).bfloat16(),
                codebook=n(V, d), r_prev=n(B, hp * wp, d), hp=hp, wp=wp, w_in=n(C, d, std=d ** -0.5), b_in=n(C, std=0.02),
                pos=n(case["h2"] * case["w2"], C, std=0.5))


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    if s["kind"] == "schedule":
        ctx = s["ctx"]
        ctx.reset()
        step = ctx.var_step_host if s["host"] else ctx.var_step
        for i, (x, keep, out) in enumerate(zip(s["maps"], s["keep"], s["outs"])):
            if s["host"]:
                step(x, i, keep, out)
            else:
                step(x, i, keep, out=out)
        if s["host"]:                            # the caller reads the maps on the host
            ctx.host_io_flush()
            torch.cuda.current_stream().synchronize()
        return s["outs"]
    if s["kind"] == "select":
        got = fv.fv_prune_select(s["x"], s["h"], s["w"], s["keep"], want_score=True, workspace=s["ws"])
        return {"idx": got["idx"], "inv": got["inv"], "score": got["score"]}
    if s["kind"] == "restore":
        return fv.fv_restore(s["cache"], s["hc"], s["wc"], s["pivots"], s["idx"], s["h"], s["w"], out=s["out"], interp_mode=s["interp"])
    ids, logits = fv.fv_head_tokens(s["y"], s["mod_head"], s["w_head"], s["b_head"], want_logits=True)
    r = fv.fv_residual_accumulate(ids, s["h"], s["w"], s["codebook"], s["r_prev"], s["hp"], s["wp"])
    return {"ids": ids, "logits": logits, "r": r, "next": fv.fv_next_scale_input(r, s["h"], s["w"], s["h2"], s["w2"], s["w_in"], s["b_in"], s["pos"])}
