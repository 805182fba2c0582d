"""The work a user of this library has it do, as cases that can be timed and whose outputs can be compared.

Four kinds of pass, each through the public entry points of `paper_2601_19139_b200.binding`:

  decode    requests join, a few decode steps run, the requests leave (the body of the serving loop).  `feed` says how
            tokens travel: "host" (decode_step_host: the serving loop reads every token before the next step),
            "device" (decode_step_chained: tokens stay on the device), "sampled" (decode_step_sampled with per-request
            temperature / top-k / top-p and given tokens).
  prefill   prompt processing of one request; `cached` tokens already have K, V (a prefix-cache hit), 0 for none.
  sample    temperature / top-k / top-p over given logits.

Models are the shapes of `workload.shapes` (0.6B, 3B, 8B, 30B-class mixture of experts) at full depth, batches 1..16,
caches of 128..8192 tokens.

What the random weights keep of trained ones: projections have unit gain, the two projections that write to the
residual stream are scaled down with depth (so that the stream stays a sum of comparable terms), and the head prefers
one token clearly (here: a fixed successor of the token fed in), so that greedy tokens are not decided by rounding.
Rows of a projection come from a bank of quantised Gaussian rows, each with a gain of its own; embedding rows are all
different.
"""
import math

import numpy as np
import torch

from paper_2601_19139_b200 import binding as B
from workload import gen, shapes

BLOCK = gen.BLOCK_SIZE
MODELS = {"0.6b": shapes.QWEN3_0P6B, "3b": shapes.LLAMA32_3B, "8b": shapes.QWEN3_8B, "moe": shapes.MOE_30B}
EMBED_STD = 0.02


def listed():
    def decode(name, model, batch, kv_lo, kv_hi, spread, steps, feed):
        return dict(name=name, kind="decode", model=model, batch=batch, kv_lo=kv_lo, kv_hi=kv_hi, spread=spread, steps=steps, feed=feed)

    def prefill(name, model, prompt, cached):
        return dict(name=name, kind="prefill", model=model, prompt=prompt, cached=cached)

    return [
        # one user chatting with the smallest model: the latency of a step, token read back each time
        decode("decode 0.6b b1 host", "0.6b", 1, 256, 256, "uniform", 4, "host"),
        # the smallest model under a full batch
        decode("decode 0.6b b16", "0.6b", 16, 128, 2048, "uniform", 4, "device"),
        # the 3B shape in the middle of its batch sweep, with sampling instead of greedy tokens
        decode("decode 3b b8 sampled", "3b", 8, 512, 4096, "uniform", 4, "sampled"),
        # the headline: 8B shape, full batch, very ragged caches
        decode("decode 8b b16", "8b", 16, 256, 8192, "log", 4, "device"),
        # an odd batch of the 8B shape in a serving loop that reads every token
        decode("decode 8b b5 host", "8b", 5, 300, 3000, "log", 4, "host"),
        # mixture of experts: full batch, and a single user
        decode("decode moe b16", "moe", 16, 512, 4096, "uniform", 4, "device"),
        decode("decode moe b1 host", "moe", 1, 1000, 1000, "uniform", 4, "host"),
        # prompts: a short chat turn, a long document, a turn that resumes after a cached prefix in the middle of a
        # block, and a mixture-of-experts prompt
        prefill("prefill 0.6b 77", "0.6b", 77, 0),
        prefill("prefill 8b 2048", "8b", 2048, 0),
        prefill("prefill 3b 2005+996", "3b", 3001, 2005),
        prefill("prefill moe 500", "moe", 500, 0),
        # the sampler alone, as a loop with its own logits processors calls it
        dict(name="sample 16x151936", kind="sample", vocab=151936, batch=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 7 + ["prefill"] * 4 + ["sample"])
    if kind == "sample":
        return dict(kind="sample", vocab=rng.choice([128256, 151936, _log_int(rng, 8000, 151936)]), batch=rng.randint(1, 16))
    model = rng.choice(sorted(MODELS))
    if kind == "prefill":
        # no more new tokens than the largest listed prompts have
        new = _log_int(rng, 17, 640 if model == "moe" else 2048)
        cached = rng.choice([0, 0, _log_int(rng, 16, 4096)])
        return _State(kind="prefill", model=model, prompt=new + cached, cached=cached)
    lo = _log_int(rng, 128, 4096)
    hi = min(8192, _log_int(rng, lo, 4 * lo))
    return dict(kind="decode", model=model, batch=_log_int(rng, 1, 16), kv_lo=lo, kv_hi=hi, spread=rng.choice(["uniform", "log"]),
                steps=rng.randint(2, 6), feed=rng.choice(["host", "device", "device", "sampled"]))


# ------------------------------------------------------------------ sizes

def _lengths(case):
    """Cached tokens of each request: evenly spread over the range (or over its logarithm)."""
    n, lo, hi = case["batch"], case["kv_lo"], case["kv_hi"]
    at = [(i + 0.5) / n for i in range(n)]
    if case["spread"] == "log":
        return [int(round(math.exp(math.log(lo) + f * math.log(hi / lo)))) for f in at]
    return [int(round(lo + f * (hi - lo))) for f in at]


def _blocks(tokens):
    return (tokens + BLOCK - 1) // BLOCK


def _layer_params(sh, experts):
    """Weights of one layer's projections that are used when `experts` experts are (dense: all)."""
    p = sh.qkv_out * sh.hidden + sh.hidden * sh.n_q_heads * sh.head_dim
    return p + (experts * 3 * sh.expert_inter * sh.hidden if sh.n_experts else 3 * sh.mlp_inter * sh.hidden)


def work(case):
    if case["kind"] == "sample":
        return {"bytes": 4.0 * case["vocab"] * case["batch"], "flops": 0.0}
    sh = MODELS[case["model"]]
    L, head = sh.n_layers, sh.vocab * sh.hidden
    heads = 4.0 * sh.n_q_heads * sh.head_dim  # multiply-adds of q k and p v per cached token, two flops each
    touched = lambda tokens: sh.n_experts * (1 - (1 - sh.top_k / sh.n_experts) ** tokens) if sh.n_experts else 0  # noqa: E731
    if case["kind"] == "prefill":
        new, start = case["prompt"] - case["cached"], case["cached"]
        weights = shapes.weight_bytes(sh, touched(new))
        kv = case["prompt"] * sh.kv_bytes_per_token
        pairs = new * start + new * (new + 1) / 2
        return {"bytes": weights + kv + 4.0 * sh.vocab,
                "flops": 2.0 * (new * L * _layer_params(sh, sh.top_k) + head) + L * heads * pairs}
    n, steps = case["batch"], case["steps"]
    kv = sum(sum(l + 1 + i for i in range(steps)) for l in _lengths(case))
    return {"bytes": steps * shapes.weight_bytes(sh, touched(n)) + kv * sh.kv_bytes_per_token + 4.0 * steps * n * sh.vocab,
            "flops": 2.0 * steps * n * (L * _layer_params(sh, sh.top_k) + head) + L * heads * kv}


def tolerance(case):
    if case["kind"] == "sample":
        return "exact"
    # every tensor between two operations is bf16: 2^-9 per rounding, over up to a hundred residual additions; two
    # correct orders of summation are 0.010..0.015 apart in the logits (0.017 with experts: near-ties of the router)
    return {"rel": 0.025 if case["model"] == "moe" else 0.02, "max": 0.4, "differ": 0.0}


# ------------------------------------------------------------------ models

def _rand(g, *size):
    return torch.rand(*size, generator=g, device="cuda")


def _projection(g, N, K, std, bank_rows=4096, gain=None):
    """A quantised [N][K] projection of standard deviation std whose rows are drawn from a bank of quantised rows."""
    w = torch.randn(bank_rows, K, generator=g, device="cuda")
    q, s, b = gen.quantize_q4(w)
    row = torch.randint(0, bank_rows, (N,), generator=g, device="cuda")
    gain = std * (0.8 + 0.4 * _rand(g, N, 1)) * (1.0 if gain is None else gain)
    return q[row], (s[row].float() * gain).to(torch.bfloat16), (b[row].float() * gain).to(torch.bfloat16)


def _norm(g, n, mean=1.0):
    return (mean + 0.02 * torch.randn(n, generator=g, device="cuda")).to(torch.bfloat16)


def _weights(sh, g):
    H, D, L = sh.hidden, sh.head_dim, sh.n_layers
    unit = lambda K: K ** -0.5  # noqa: E731
    branch = 1.5 * EMBED_STD / math.sqrt(2 * L)
    sharp = 1.5  # how far attention logits spread
    q_gain = torch.ones(sh.qkv_out, 1, device="cuda")
    if not sh.qk_norm:
        q_gain[:sh.n_q_heads * D] = sharp
    layers = []
    for _ in range(L):
        lw = {"attn_norm": _norm(g, H), "mlp_norm": _norm(g, H),
              "q_norm": _norm(g, D, sharp) if sh.qk_norm else None, "k_norm": _norm(g, D) if sh.qk_norm else None,
              "wqkv": _projection(g, sh.qkv_out, H, unit(H), gain=q_gain),
              "wo": _projection(g, H, sh.n_q_heads * D, branch * unit(sh.n_q_heads * D))}
        if sh.n_experts:
            E, I = sh.n_experts, sh.expert_inter
            lw["router"] = (2.5 * unit(H) * torch.randn(E, H, generator=g, device="cuda")).to(torch.bfloat16)
            lw["experts_gate_up"] = _projection(g, E * 2 * I, H, unit(H))
            lw["experts_down"] = _projection(g, E * H, I, branch * unit(I))
        else:
            lw["w_gate_up"] = _projection(g, 2 * sh.mlp_inter, H, unit(H))
            lw["w_down"] = _projection(g, H, sh.mlp_inter, branch * unit(sh.mlp_inter))
        layers.append(lw)
    parts = [gen.quantize_q4(EMBED_STD * torch.randn(min(16384, sh.vocab - r), H, generator=g, device="cuda"))
             for r in range(0, sh.vocab, 16384)]
    embed = tuple(torch.cat(p) for p in zip(*parts))
    lm_head = embed
    if not sh.tie_embeddings:
        order = torch.randperm(sh.vocab, generator=g, device="cuda")
        lm_head = tuple(t[order] for t in embed)
    return {"layers": layers, "final_norm": _norm(g, H), "embed": embed, "lm_head": lm_head,
            "rope": _rope(sh)}


_ROPE = {}


def _rope(sh):
    """The rotary table, a constant of the model family."""
    key = (sh.max_positions, sh.head_dim, sh.rope_base)
    if key not in _ROPE:
        _ROPE[key] = gen.rope_table(*key, device="cuda")
    return _ROPE[key]


def _pool(sh, g, num_blocks):
    """Prefilled K, V: values that have a mean of their own per channel, as cached states have."""
    pool = torch.empty(gen.pool_shape(sh, num_blocks), dtype=torch.bfloat16, device="cuda")
    for layer in pool:
        layer.normal_(generator=g)
        layer[1] += 0.5 * torch.randn(1, sh.n_kv_heads, 1, sh.head_dim, generator=g, device="cuda", dtype=torch.bfloat16)
    return pool


# ------------------------------------------------------------------ a pass

class _State(dict):
    """What a pass needs; the library's objects go with it."""

    def __del__(self):
        for key in ("pool", "model"):
            if key in self:
                self[key].close()


def _shuffled(order, first, count):
    """`count` block ids from `first` on, in random order (block tables are never contiguous in a pool that has lived)."""
    return first + order.permutation(count).astype(np.int32)


def _prepare_decode(case, sh, g, order):
    n, steps, lens = case["batch"], case["steps"], _lengths(case)
    order.shuffle(lens)
    first_new = [l // BLOCK for l in lens]
    need = [_blocks(l + steps) for l in lens]
    written = sum(b - a for a, b in zip(first_new, need))  # blocks that receive new tokens: ids 0..written-1
    total = sum(need)
    new_ids, old_ids = list(_shuffled(order, 0, written)), list(_shuffled(order, written, total - written))
    tables = np.zeros((n, max(need)), dtype=np.int32)
    for r in range(n):
        for i in range(need[r]):
            tables[r, i] = (new_ids if i >= first_new[r] else old_ids).pop()
    model = B.Model(sh, _weights(sh, g))
    pool = B.KVPool(model, _pool(sh, g, total))
    st = _State(kind="decode", feed=case["feed"], steps=steps, model=model, pool=pool, ids=np.arange(n, dtype=np.int64) + 1,
              lens=lens, tables=tables, updated=pool.mem[:, :, :written],
              tokens=order.integers(0, sh.vocab, n).astype(np.int32),
              next=torch.zeros(steps, n, dtype=torch.int32, device="cuda"),
              logits=torch.zeros(n, sh.vocab, dtype=torch.float32, device="cuda"))
    st["tokens_device"] = torch.from_numpy(st["tokens"]).cuda()
    if case["feed"] == "sampled":
        st["given"] = order.integers(0, sh.vocab, (steps, n)).astype(np.int32)
        st["sampling"] = (order.uniform(0.3, 0.8, n).astype(np.float32), order.choice([0, 20, 50, 200], n).astype(np.int32),
                          order.choice([0.8, 0.9, 0.95, 1.0], n).astype(np.float32))
        st["u"] = order.uniform(0, 1, (steps, n)).astype(np.float32)
    return st


def _prepare_prefill(case, sh, g, order):
    prompt, cached = case["prompt"], case["cached"]
    need, first_new = _blocks(prompt), cached // BLOCK
    written = need - first_new
    table = np.concatenate([_shuffled(order, written, first_new), _shuffled(order, 0, written)]).astype(np.int32)
    model = B.Model(sh, _weights(sh, g))
    pool = B.KVPool(model, _pool(sh, g, need))
    return _State(kind="prefill", model=model, pool=pool, cached=cached, table=table, updated=pool.mem[:, :, :written],
                tokens=order.integers(0, sh.vocab, prompt).astype(np.int32),
                next=torch.zeros(1, dtype=torch.int32, device="cuda"),
                logits=torch.zeros(sh.vocab, dtype=torch.float32, device="cuda"))


def _prepare_sample(case, g, order):
    n, V = case["batch"], case["vocab"]
    # a language model's next-token logits: a broad body, and a few hundred candidates that carry the probability
    logits = 2.0 * torch.randn(n, V, generator=g, device="cuda")
    top = torch.randint(0, V, (n, 300), generator=g, device="cuda")
    logits.scatter_(1, top, 8.0 + 8.0 * _rand(g, n, 300) ** 2)
    sampling = (order.uniform(0.5, 1.2, n).astype(np.float32), order.choice([0, 20, 50, 200], n).astype(np.int32),
                order.choice([0.8, 0.9, 0.95, 1.0], n).astype(np.float32), order.uniform(0, 1, n).astype(np.float32))
    return dict(kind="sample", logits=logits, sampling=sampling)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    order = np.random.default_rng(seed)
    if case["kind"] == "sample":
        return _prepare_sample(case, g, order)
    sh = MODELS[case["model"]]
    return (_prepare_decode if case["kind"] == "decode" else _prepare_prefill)(case, sh, g, order)


def _run_decode(st):
    model, pool, ids, tables = st["model"], st["pool"], st["ids"], st["tables"]
    for rid, length in zip(ids.tolist(), st["lens"]):
        pool.request_admit(rid, length)
    out = {"kv": st["updated"]}
    if st["feed"] == "host":
        tokens, got = st["tokens"], []
        for _ in range(st["steps"]):
            tokens, _unused = B.decode_step_host(model, pool, ids, tokens, tables)
            got.append(tokens)
        out["tokens"] = np.stack(got)
    elif st["feed"] == "device":
        tokens = st["tokens_device"]
        for i in range(st["steps"]):
            last = i == st["steps"] - 1
            B.decode_step_chained(model, pool, ids, tokens, tables, st["next"][i], st["logits"] if last else None)
            tokens = st["next"][i]
        out["tokens"], out["logits"] = st["next"], st["logits"]
    else:
        for i in range(st["steps"]):
            B.decode_step_sampled(model, pool, ids, st["given"][i], tables, *st["sampling"], st["u"][i], st["next"][i], st["logits"])
        out["tokens"], out["logits"] = st["next"], st["logits"]
    for rid in ids.tolist():
        pool.request_release(rid)
    return out


def run(state):
    if state["kind"] == "decode":
        return _run_decode(state)
    if state["kind"] == "prefill":
        B.prefill(state["model"], state["pool"], 1, state["tokens"], state["cached"], state["table"], state["next"], state["logits"])
        state["pool"].request_release(1)
        return {"kv": state["updated"], "token": state["next"], "logits": state["logits"]}
    return {"tokens": B.sample(state["logits"], *state["sampling"])}
