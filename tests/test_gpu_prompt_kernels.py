"""Prompt processing at the edges of its kernels' tiles, against the oracle: token tiles (16-multiples up to 256), key
tiles of 64, partly filled blocks, operand widths whose group sums fill a stage partly, experts with no and many tokens."""
import numpy as np
import pytest
import torch

from oracle import q4d_oracle as orc
from workload import gen, shapes


def _dense(**kw):
    a = dict(n_layers=1, hidden=256, n_q_heads=4, n_kv_heads=2, mlp_inter=256, vocab=512, max_positions=1024)
    a.update(kw)
    return shapes.toy("prompt-toy-" + "-".join(f"{k}{v}" for k, v in sorted(kw.items())), **a)


def _moe(n_experts, top_k):
    return shapes.toy(f"prompt-toy-moe{n_experts}", n_layers=1, hidden=256, n_q_heads=4, n_kv_heads=2, mlp_inter=256, vocab=512,
                      n_experts=n_experts, top_k=top_k, expert_inter=256, norm_topk_prob=1, max_positions=1024)


MOE = _moe(12, 3)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,n_tokens,start", [
    (_dense(), 17, 0), (_dense(), 64, 0), (_dense(), 65, 0), (_dense(), 257, 0), (_dense(), 130, 77), (_dense(), 97, 80),
    (_dense(hidden=1024, n_q_heads=8, n_kv_heads=1), 33, 0),          # 16 groups: one full stage of sums; 8 heads per kv head
    (_dense(hidden=1280, mlp_inter=2304), 40, 0),                     # 20 and 36 groups: partly filled stages
    (_dense(qk_norm=0, n_q_heads=6, mlp_inter=768), 50, 16),
    (MOE, 17, 0), (MOE, 150, 0), (MOE, 61, 32),
    (_moe(80, 8), 70, 0), (_moe(144, 2), 33, 0),                      # the router's features in two parts, and in one
], ids=lambda v: getattr(v, "name", str(v)))
def test_prompt_kernels_at_tile_edges(shape, n_tokens, start):
    from gpu_util import bits, from_bits
    from paper_2601_19139_b200 import binding as q4d
    weights, pool_t = gen.make_weights(shape, 5, "cuda"), gen.make_pool(shape, 24, "cuda")
    om = orc.OracleModel(shape, weights)
    rng = np.random.default_rng(1000 + n_tokens)
    prompt = rng.integers(0, shape.vocab, size=n_tokens).astype(np.int32)
    table = [int(b) for b in rng.permutation(np.arange(1, 24))[:(n_tokens + 15) // 16]]
    host = orc.to_np(pool_t).copy()
    if start:
        orc.prefill(om, host, 16, prompt[:start], 0, table)
        for b in table[:(start + 15) // 16]:
            pool_t[:, :, b] = from_bits(host[:, :, b])
    before = bits(pool_t)
    o_next, o_logits = orc.prefill(om, host, 16, prompt, start, table)
    model = q4d.Model(shape, weights)
    pool = q4d.KVPool(model, pool_t)
    nxt = torch.zeros(1, dtype=torch.int32, device="cuda")
    lg = torch.zeros(shape.vocab, dtype=torch.float32, device="cuda")
    for _ in range(2):   # the second run finds the counters and buffers the first one left
        q4d.prefill(model, pool, 7, prompt, start, table, nxt, lg)
        pool.request_release(7)
    torch.cuda.synchronize()
    got = bits(pool_t)
    for t in range(n_tokens):
        where = (slice(None), slice(None), table[t // 16], slice(None), t % 16)
        if t < start:
            assert np.array_equal(got[where], before[where])
        else:
            g, w = orc.bf16_to_f64(got[where]), orc.bf16_to_f64(host[where])
            rms = np.sqrt((w ** 2).mean())
            assert np.sqrt(((g - w) ** 2).mean()) <= 6e-3 * rms and np.abs(g - w).max() <= 0.1 * rms, t
    assert np.array_equal(got[:, :, 0], before[:, :, 0])
    g = lg.cpu().numpy().astype(np.float64)
    rms = np.sqrt((o_logits.astype(np.float64) ** 2).mean())
    assert np.abs(g - o_logits).max() <= (0.15 if shape.n_experts else 3e-2) * rms
    pool.close()
    model.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape,n_tokens", [(_dense(hidden=2048, mlp_inter=6144, n_layers=2), 1000), (_dense(hidden=3072, mlp_inter=4096), 760),
                                            (_moe(24, 8), 1000)], ids=lambda v: getattr(v, "name", str(v)))
def test_wide_tiles_repeat_bit_for_bit(shape, n_tokens):
    """Several tiles per CTA, so that the rings of codes and operands turn many times: any order of the warps gives the same."""
    from gpu_util import bits
    from paper_2601_19139_b200 import binding as q4d
    weights, pool_t = gen.make_weights(shape, 5, "cuda"), gen.make_pool(shape, 64, "cuda")
    model = q4d.Model(shape, weights)
    pool = q4d.KVPool(model, pool_t)
    prompt = np.random.default_rng(3).integers(0, shape.vocab, size=n_tokens).astype(np.int32)
    table = list(range(1, 1 + (n_tokens + 15) // 16))
    lg = torch.zeros(shape.vocab, dtype=torch.float32, device="cuda")
    seen = []
    for _ in range(6):
        q4d.prefill(model, pool, 7, prompt, 0, table, None, lg)
        pool.request_release(7)
        torch.cuda.synchronize()
        seen.append((bits(pool_t)[:, :, table].copy(), lg.cpu().numpy().copy()))
    for kv, logits in seen[1:]:
        assert np.array_equal(kv, seen[0][0]) and np.array_equal(logits, seen[0][1])
