"""Inputs that a kernel of the library has just written on the stream.  A launch may start while the kernels before it still run
(programmatic dependent launch), so whatever it reads before its dependency wait can be stale.  Producer and consumer are replayed
from one CUDA graph, back to back, over a buffer that held other values; the consumer's result has to be the one it gives when the buffer
is at rest."""
import numpy as np
import pytest
import torch

from paper_2503_23367_b200 import binding as fv
from paper_2503_23367_b200 import inputs as I

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


def _check_in_order(produce, consume, renew, rounds=4):
    """consume() -> a tensor or a list of them."""
    as_list = lambda v: list(v) if isinstance(v, (list, tuple)) else [v]
    renew(0)
    produce()
    consume()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        produce()
        got = as_list(consume())
    for i in range(1, rounds + 1):
        renew(i)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        mine = [t.clone() for t in got]
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
