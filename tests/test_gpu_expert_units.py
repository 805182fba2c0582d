"""Routed experts where their units can go wrong: an expert with more than 8 of the 16 requests, expert counts that are no
multiple of 8, one request, a single expert for everybody, the widest list of units."""
import numpy as np
import pytest
import torch

from gpu_util import Scenario, bits
from oracle import q4d_oracle as orc
from workload import shapes

LENS = [3, 100, 31, 64, 9, 200, 1, 0, 22, 50, 12, 47, 8, 63, 15, 16]


def _shape(E, k, hidden=256, inter=256):
    return shapes.toy(f"units-{E}-{k}-{hidden}-{inter}", n_layers=1, hidden=hidden, n_q_heads=4, n_kv_heads=2, mlp_inter=256, vocab=512,
                      n_experts=E, top_k=k, expert_inter=inter, norm_topk_prob=1)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,n", [(_shape(1, 1), 16), (_shape(3, 2), 16), (_shape(12, 7), 9), (_shape(20, 32 - 12, 512, 768), 16),
                                     (_shape(256, 32), 16), (_shape(130, 4, 768, 512), 1)], ids=lambda v: getattr(v, "name", str(v)))
def test_layer_with_uneven_units(shape, n):
    from paper_2601_19139_b200 import binding as q4d
    sc = Scenario(shape, LENS[:n], seed=6)
    bt = sc.block_tables()
    _, _, taps = sc.oracle.decode_step(sc.host_pool.copy(), 16, sc.lens, sc.tokens, bt, want_taps=True)
    model = q4d.Model(shape, sc.weights)
    pool = q4d.KVPool(model, sc.pool)
    ids = np.arange(n, dtype=np.int64)
    for r in range(n):
        pool.request_admit(int(ids[r]), sc.lens[r])
    x0 = q4d.embed(sc.weights["embed"], torch.from_numpy(sc.tokens).cuda())
    for _ in range(2):   # the second run finds the counters the first one left
        got = q4d.debug_run_layers(model, pool, ids, bt, 0, 1, x0)
    g, w = orc.bf16_to_f64(bits(got)), orc.bf16_to_f64(taps[1])
    err = np.sqrt(((g - w) ** 2).mean(-1) / (w ** 2).mean(-1))
    assert np.sort(err)[-2 if n > 1 else -1] <= 6e-3 and err.max() <= 0.1, err   # a near-tie of the router may move one request
    assert model.moe_touched_experts() >= 0
    pool.close()
    model.close()
