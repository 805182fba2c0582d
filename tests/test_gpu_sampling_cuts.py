"""The sampler where its cuts do not fit the sorted list, and at the smallest and largest slices of the vocabulary."""
import numpy as np
import pytest
import torch

from oracle import q4d_oracle as orc


@pytest.mark.gpu
@pytest.mark.parametrize("V,distinct,T,k,p", [
    (1, 1, 1.0, 0, 1.0), (7, 7, 1.0, 3, 0.9), (8 * 4096, 1, 1.0, 0, 1.0),      # one logit shared by all
    (40000, 3, 1.0, 20000, 0.7), (40000, 3, 1.0, 0, 0.5), (40000, 2, 0.7, 0, 1.0),  # few values, thousands of ties each
    (30000, 30000, 4.0, 12000, 0.95), (30000, 30000, 50.0, 0, 1.0),             # flat: thousands of tokens are kept
    (300001, 300001, 1.0, 100, 0.9), (300001, 4, 1.0, 0, 0.8),                  # slices that do not fit shared memory
])
def test_sample_beyond_the_list(V, distinct, T, k, p):
    from paper_2601_19139_b200 import binding as q4d
    rng = np.random.default_rng(V + distinct + k)
    n = 5
    logits = (rng.standard_normal((n, V)) * 1.5).astype(np.float32)
    if distinct < V:
        values = np.sort(rng.standard_normal(distinct).astype(np.float32))
        logits = values[rng.integers(0, distinct, size=(n, V))]
    us = np.array([0.0, 0.25, 0.5, 0.9, 1.0 - 2.0 ** -24], dtype=np.float32)
    got = q4d.sample(torch.from_numpy(logits).cuda(), [T] * n, [k] * n, [p] * n, us).cpu().numpy()
    exact = 0
    for r in range(n):
        want = orc.sample_token(logits[r], T, k, p, float(us[r]))
        if got[r] == want:
            exact += 1
            continue
        # the weights differ by parts in 10^7 (fp32 against fp64 exponentials): the neighbour of a boundary is allowed
        order, w, kept = orc.sampling_table(logits[r], T, k, p)
        cum = np.cumsum(w[:kept].astype(np.float64))
        at = int(np.flatnonzero(order[:kept] == got[r])[0])
        t = float(us[r]) * cum[-1]
        assert (cum[at - 1] if at else 0.0) - 1e-5 * cum[-1] <= t <= cum[at] + 1e-5 * cum[-1]
    assert exact >= (n - 1 if distinct == V or distinct == 1 else 0)
