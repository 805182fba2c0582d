"""The dense projections at the edges of their split: one to sixteen K-slices per CTA, an odd last slice, K over several
CTAs, ragged last row tiles, both request counts, scales with and without tensor maps, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import q4d_oracle as orc
from workload import gen


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,n", [
    (8, 256, 1), (16, 256, 16), (200, 768, 9), (24, 512, 8), (4096 * 2 + 8, 256, 3),      # few slices, ragged rows
    (136, 3840, 16), (136, 4096, 8), (40, 4096 + 256, 16), (40, 4096 + 512, 2),            # around the slices of one CTA
    (2500, 1280, 16), (64, 12288, 5), (48, 16384, 11),                                     # odd slices; K in several parts
])
def test_projection_split_edges(N, K, n):
    from gpu_util import bits, from_bits
    from paper_2601_19139_b200 import binding as q4d
    q, s, b = gen.random_q4(N, K, "cpu", "tiles", N, K)
    g = torch.Generator().manual_seed(N + K + n)
    x = (torch.randn(n, K, generator=g) * torch.exp2(torch.randint(-6, 7, (n, K), generator=g).float())).to(torch.bfloat16)
    # fp64 definition: w = fl32(scale q + bias)
    code = (q.to(torch.int64).unsqueeze(-1) >> (4 * torch.arange(8))) & 15
    w = code.view(N, K // 64, 64).double() * s.double().unsqueeze(-1) + b.double().unsqueeze(-1)
    w = w.float().double().view(N, K)
    want = x.double() @ w.T
    dev = tuple(t.cuda() for t in (q, s, b))
    for _ in range(2):   # the second call finds the counters the first one left
        got = q4d.q4_gemm(dev, x.cuda(), n, epilogue=2)
    err = (got.cpu().double() - want).abs().max() / want.square().mean().sqrt()
    assert err <= 3e-5, float(err)
    y = q4d.q4_gemm(dev, x.cuda(), n, epilogue=0)
    assert bits(y).shape == (n, N)
    assert ((y.cpu().double() - want).abs() <= want.abs() * 2 ** -8 + 1e-4 * want.square().mean().sqrt()).all()
