"""Row kernels at the sizes where their dispatch changes: the norm's registers per row length and batch, the merge of an
attention request at the edges of its batches of chunks (8 partial results, 32 weights)."""
import numpy as np
import pytest
import torch

from oracle import q4d_oracle as orc
from workload import gen


@pytest.mark.gpu
@pytest.mark.parametrize("H", [64, 2048, 2112, 3072, 3136, 4096, 4160, 8192, 8256, 16384])
@pytest.mark.parametrize("n", [1, 8, 9, 16])
def test_norm_of_every_row_length(n, H):
    from gpu_util import assert_bf16_close, bits
    from paper_2601_19139_b200 import binding as q4d
    g = torch.Generator(device="cuda").manual_seed(H + n)
    x = (0.3 * torch.randn(n, H, generator=g, device="cuda")).to(torch.bfloat16)
    w = gen.norm_weight(H, "cuda", "row-norm", H)
    assert_bf16_close(bits(q4d.rmsnorm(x, w, 1e-6)), orc.rmsnorm(bits(x), bits(w), 1e-6), what="rmsnorm")


@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(4, 2), (24, 8), (16, 2), (16, 1)])
def test_merge_of_every_number_of_chunks(nq, nkv):
    from gpu_util import assert_bf16_close, bits
    from paper_2601_19139_b200 import binding as q4d
    chunks = [1, 2, 7, 8, 9, 16, 31, 32, 33, 40, 41, 65]
    lens = [16 * c - 1 - (c % 3) for c in chunks]       # chunks of one block; the new token is the last of each request
    g = torch.Generator(device="cuda").manual_seed(5)
    blocks = sum(chunks) + 3
    pool = torch.randn(2, blocks, nkv, 16, 128, generator=g, device="cuda").to(torch.bfloat16)
    q = torch.randn(len(lens), nq, 128, generator=g, device="cuda").to(torch.bfloat16)
    order, bt, at = np.random.default_rng(6).permutation(blocks), np.zeros((len(lens), max(chunks)), np.int32), 0
    for r, c in enumerate(chunks):
        bt[r, :c], at = order[at:at + c], at + c
    out = q4d.paged_attention(q, pool[0], pool[1], lens, torch.from_numpy(bt).cuda(), chunk_tokens=16)
    want = orc.attention_paged(bits(q), bits(pool)[None], nq, nkv, 16, 128, 0, lens, bt)
    assert_bf16_close(bits(out), want, what="attention")
