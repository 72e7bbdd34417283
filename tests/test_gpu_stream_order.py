"""Inputs that a kernel of the library has just written on the stream.  A launch may start while the kernels before it still run
(programmatic dependent launch), so whatever it reads before its dependency wait can be stale.  Producer and consumer are replayed
from one CUDA graph, back to back, over a buffer that held other values; the consumer's result has to be the one it gives when the buffer
is at rest."""
import numpy as np
import pytest
import torch

from paper_2503_23367_b200 import binding as fv

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _randn(seed, *shape, std=1.0, dtype=torch.float32):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return (torch.randn(*shape, generator=g, device=DEV) * std).to(dtype)


class _LongGemm:
    """out = A W^T over a long K into the caller's buffer, by the library's own GEMM: a producer that is still running when the
    kernel behind it starts.  Another A in every round, so that a stale buffer shows."""

    def __init__(self, rows, cols, dtype, K=8192):
        self.a = _randn(1, rows, K, dtype=torch.bfloat16)
        self.w = _randn(2, cols, K, std=0.02, dtype=torch.bfloat16)
        self.out = torch.zeros(rows, cols, dtype=dtype, device=DEV)
        self.rows, self.K = rows, K

    def renew(self, i):
        self.a.copy_(_randn(10 + i, self.rows, self.K, dtype=torch.bfloat16))
        self.out.fill_(-7.0)

    def __call__(self):
        fv.fv_gemm_bf16(self.a, self.w, None, 4 if self.out.dtype == torch.float32 else 0, out=self.out)


def _check_in_order(produce, consume, renew, rewind=lambda: None, rounds=4):
    """consume() -> a tensor or a list of them; rewind() puts back what it works on in place."""
    as_list = lambda v: list(v) if isinstance(v, (list, tuple)) else [v]
    renew(0)
    rewind()
    produce()
    consume()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        produce()
        got = as_list(consume())
    for i in range(1, rounds + 1):
        renew(i)
        rewind()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        mine = [t.clone() for t in got]
        rewind()
        want = as_list(consume())                  # the produced buffer at rest
        torch.cuda.synchronize()
        for a, b in zip(mine, want):
            assert torch.equal(a, b), f"round {i}: the consumer has read what its producer had not written yet"


@pytest.mark.parametrize("M,N,K", [(1, 2048, 2048), (32, 2048, 8192), (40, 6144, 2048), (48, 9600, 512), (100, 1024, 4096), (200, 2048, 2048), (400, 2048, 1024)])
def test_gemm_bias_written_by_the_kernel_before(M, N, K):
    bias = _LongGemm(8, N, torch.bfloat16)
    a, w = _randn(3, M, K, dtype=torch.bfloat16), _randn(4, N, K, std=0.02, dtype=torch.bfloat16)
    _check_in_order(bias, lambda: fv.fv_gemm_bf16(a, w, bias.out[0]), bias.renew)


@pytest.mark.parametrize("k,n,C", [(1, 1, 1024), (9, 256, 2048), (600, 1024, 512)])
def test_layernorm_modulation_written_by_the_kernel_before(k, n, C):
    mod = _LongGemm(2, 2 * C, torch.float32)               # two images: sigma, beta
    x = _randn(5, 2, n, C)
    idx = torch.stack([torch.randperm(n, generator=torch.Generator().manual_seed(b))[:k].sort().values for b in range(2)]).int().to(DEV)
    flat = mod.out.view(-1)
    _check_in_order(mod, lambda: fv.fv_gather_ln(x, idx, flat[:C], flat.data_ptr() + 4 * C, mod_stride=2 * C), mod.renew)


@pytest.mark.parametrize("step,keep,last", [(1, 1.0, 16), (2, 0.5, 16), (2, 0.3, 40)])
@pytest.mark.parametrize("in_place", [True, False])
def test_step_with_modulation_written_by_the_kernel_before(step, keep, last, in_place):
    """In place no copy stands in front of the step's first kernel: gather + LayerNorm (unpruned), the one-launch selection of a small map,
    the selection of a larger one.  Out of place one does, and the kernels behind it may read the modulation before their own waits."""
    L, B, C, H = 2, 2, 256, 4
    sides = [(2, 2), (8, 8), (last, last)]
    g = torch.Generator(device=DEV)
    g.manual_seed(3)

    def w(*shape):
        return [(torch.randn(*shape, generator=g, device=DEV) * 0.02).bfloat16() for _ in range(L)]

    class Tensors:
        w_qkv, b_qkv, w_o, b_o = w(3 * C, C), w(3 * C), w(C, C), w(C)
        w_fc1, b_fc1, w_fc2, b_fc2 = w(4 * C, C), w(4 * C), w(C, 4 * C), w(C)
        w_q_x = w_kv_x = w_o_x = text = None
        mod = torch.randn(L, B, 6, C, generator=g, device=DEV) * 0.3

    ctx = fv.FvContext(L, C, H, sides, 1, B, 4 + 64 + last * last, Tensors)
    produce = _LongGemm(L * B, 6 * C, torch.float32)
    produce.out = ctx.mod.view(L * B, 6 * C)
    maps = [_randn(20 + i, B, a * b, C) for i, (a, b) in enumerate(sides)]
    for i, m in enumerate(maps):                       # fills the caches and the keys of the steps before
        ctx.var_step(m, i, keep if i == 2 else 1.0)
    x = maps[step].clone()
    kv = sum(a * b for a, b in sides[:step])

    def consume():
        ctx.set_state(step, kv)
        return ctx.var_step(x, step, keep, out=x if in_place else None).clone()

    _check_in_order(produce, consume, produce.renew, rewind=lambda: x.copy_(maps[step]))
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("d", [8, 32, 64])
def test_next_token_map_with_w_in_written_by_the_kernel_before(d):
    C = 512
    w_in = _LongGemm(C, d, torch.float32)
    r, b_in, pos = _randn(6, 2, 36, d), _randn(7, C), _randn(8, 64, C)
    _check_in_order(w_in, lambda: fv.fv_next_scale_input(r, 6, 6, 8, 8, w_in.out, b_in, pos), w_in.renew)


class _Selection:
    """The library's selection into the caller's buffers, on a map that changes from round to round."""

    def __init__(self, B, h, w, C, keep):
        self.B, self.h, self.w, self.C, self.keep = B, h, w, C, keep
        self.k = fv.fv_k_for(keep, h, w)
        self.x = torch.empty(B, h * w, C, device=DEV)
        self.idx = torch.zeros(B, self.k, dtype=torch.int32, device=DEV)
        self.ws = fv.fv_prune_select_workspace(B, h * w, C, DEV)

    def renew(self, i):
        self.x.copy_(_randn(40 + i, self.B, self.h * self.w, self.C))
        self.idx.copy_(torch.arange(self.k, dtype=torch.int32, device=DEV).expand(self.B, -1))

    def __call__(self):
        rc = fv.lib().fv_prune_select(self.x.data_ptr(), self.B, self.h, self.w, self.C, self.keep, self.idx.data_ptr(), None, None, None, None,
                                      self.ws.data_ptr(), self.ws.numel(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0


@pytest.mark.parametrize("B,h,w,C,keep", [(2, 12, 12, 256, 0.4), (1, 64, 64, 2048, 0.2)])
@pytest.mark.parametrize("interp", [0, 1, 2])
def test_restoration_of_indices_written_by_the_kernel_before(B, h, w, C, keep, interp):
    sel = _Selection(B, h, w, C, keep)
    cache, pivots = _randn(50, B, (h // 2) * (w // 2), C, dtype=torch.bfloat16), _randn(51, B, sel.k, C, dtype=torch.bfloat16)
    _check_in_order(sel, lambda: fv.fv_restore(cache, h // 2, w // 2, pivots, sel.idx, h, w, interp_mode=interp), sel.renew)


def test_gather_of_indices_written_by_the_kernel_before():
    sel = _Selection(2, 40, 40, 1024, 0.3)
    _check_in_order(sel, lambda: fv.fv_gather_ln(sel.x, sel.idx, None, None), sel.renew)


def test_restoration_of_rows_written_by_the_kernel_before():
    B, h, w, C, k = 2, 12, 12, 512, 48
    pivots = _LongGemm(B * k, C, torch.bfloat16)
    cache = _randn(52, B, 36, C, dtype=torch.bfloat16)
    idx = torch.arange(0, 3 * k, 3, dtype=torch.int32, device=DEV).expand(B, -1).contiguous()
    _check_in_order(pivots, lambda: fv.fv_restore(cache, 6, 6, pivots.out.view(B, k, C), idx, h, w), pivots.renew)


def test_residual_and_next_map_of_tokens_written_by_the_kernel_before():
    """Head logits -> ids -> Eq. 2 -> next map, each kernel the producer of the next."""
    B, h, w, V, d, C = 2, 16, 16, 1024, 32, 512
    logits = _LongGemm(B * h * w, V, torch.float32, K=2048)
    codebook, r_prev, w_in = _randn(60, V, d), _randn(61, B, 64, d), _randn(62, C, d)

    def consume():
        ids = fv.fv_argmax_rows(logits.out).view(B, h * w)
        r = fv.fv_residual_accumulate(ids, h, w, codebook, r_prev, 8, 8)
        return ids, r, fv.fv_next_scale_input(r, h, w, 20, 20, w_in, None, None)

    _check_in_order(logits, consume, logits.renew)
