"""The work that users of this library have it do, as measurable cases.

A case names one use of the public entry points with its sizes: a draft+verify round of a whole model (`round`), a chunk
of prompt through the same step (`prefill`), rounds that stay on the device (`device_rounds`), and the operations that
another engine calls by themselves: greedy verification of given logits (`verify`), the hybrid-mask paged attention of a
whole forward (`attention`), and moving the K/V of a request into or out of the pool (`kv_write`, `kv_read`).  Shapes, block
sizes and context ranges are those of the package's configurations, tests and benchmark.

The lengths of a batch follow from the case alone (`batch` seeds them); weights, tokens and K/V follow from `prepare`'s seed.

Weights.  Random weights of the plain recipe make a model whose logits carry no information: its top tokens are near ties,
which rounding decides.  Two things that trained models have are therefore added.  The projections that write the residual
stream are scaled by 1/sqrt(2 n_layers) (the usual depth-scaled initialisation), with embeddings of unit scale, so that
rounding errors do not pile up over the depth.  And the LM head knows a successor of every token, so that the verifier
prefers one token clearly and planted drafts are accepted or rejected by it as in real decoding.
"""
import math

import numpy as np
import torch

from paper_2609_34388_b200 import binding, synth

PAGE = 16


# ---- shapes -----------------------------------------------------------------------------------------------------------
def _shape(case):
    name = case["model"]
    if name == "tiny":
        return synth.tiny_shape()                       # head_dim 64
    if name == "small":                                 # the smallest model with head_dim 128
        return synth.ModelShape(n_layers=2, hidden=512, n_q_heads=4, n_kv_heads=2, head_dim=128, ffn=1024, vocab=2048)
    if name == "14b":
        return synth.dense14b_shape()                   # five query heads per kv head
    return synth.llama8b_shape()


def listed():
    return [
        # the smallest round: launches and latency are all there is
        {"name": "round_tiny_3", "op": "round", "model": "tiny", "n_req": 3, "blocks": "4,8", "ctx_lo": 20, "ctx_hi": 200,
         "branches": 0, "logits": "f32", "host": True, "batch": 3},
        # one user, low latency: 16 verify rows and 16 mask rows over 4096 tokens of context, results needed on the host
        {"name": "round_8b_1", "op": "round", "model": "8b", "n_req": 1, "blocks": "16", "ctx_lo": 4096, "ctx_hi": 4096,
         "branches": 0, "logits": "f32", "host": True, "batch": 3},
        # a few users of the larger model
        {"name": "round_14b_4", "op": "round", "model": "14b", "n_req": 4, "blocks": "8,16", "ctx_lo": 512, "ctx_hi": 4096,
         "branches": 0, "logits": "f32", "host": True, "batch": 3},
        # the ordinary serving batch
        {"name": "round_8b_16", "op": "round", "model": "8b", "n_req": 16, "blocks": "4,8,16,32", "ctx_lo": 512,
         "ctx_hi": 8192, "branches": 0, "logits": "f32", "host": True, "batch": 3},
        # predictive overlap: two correction branches per request
        {"name": "round_8b_8_branches", "op": "round", "model": "8b", "n_req": 8, "blocks": "8,16,32", "ctx_lo": 512,
         "ctx_hi": 8192, "branches": 2, "logits": "f32", "host": True, "batch": 5},
        # high load: small blocks, many requests, bf16 logits, results consumed on the device
        {"name": "round_8b_128", "op": "round", "model": "8b", "n_req": 128, "blocks": "2,4,8,16", "ctx_lo": 256,
         "ctx_hi": 3072, "branches": 0, "logits": "bf16", "host": False, "batch": 3},
        # two prompts in chunks of about a thousand tokens, one of them far into its context
        {"name": "prefill_8b_2048", "op": "prefill", "model": "8b", "n_req": 2, "chunk_lo": 900, "chunk_hi": 1024, "ctx_lo": 0,
         "ctx_hi": 6000, "batch": 4},
        # rounds that never wait for the host: block sizes by the rule, acceptance lengths from the planted chain
        {"name": "device_rounds_8b_4", "op": "device_rounds", "model": "8b", "n_req": 4, "rounds": 4, "block": 16,
         "ctx_lo": 512, "ctx_hi": 4096, "batch": 3},
        # verification of another engine's logits: one request with four drafts, and a large batch that drafts as well
        {"name": "verify_5_rows", "op": "verify", "n_req": 1, "drafts": 4, "block": 0, "vocab": 128256, "logits": "f32", "host": True},
        {"name": "verify_8448_rows", "op": "verify", "n_req": 256, "drafts": 16, "block": 16, "vocab": 128256, "logits": "bf16",
         "host": True},
        # the attention of one forward for another engine's model: one request, all layers
        {"name": "attention_8b_1", "op": "attention", "model": "8b", "n_req": 1, "blocks": "16", "ctx_lo": 4096,
         "ctx_hi": 4096, "branches": 0, "batch": 3},
        # a prefix computed elsewhere comes into the pool, all layers
        {"name": "kv_write_8b_4001", "op": "kv_write", "model": "8b", "n_pos": 4001, "pos0": 0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["round", "round", "round", "round", "prefill", "device_rounds", "verify", "attention", "kv_write", "kv_read"])
    batch = rng.randrange(1, 1 << 20)
    if op in ("round", "attention"):
        model = rng.choice(["8b", "8b", "8b", "14b", "tiny", "small"] if op == "round" else ["8b", "8b", "14b"])
        n_req = _log_int(rng, 1, 12 if model == "14b" else (128 if op == "round" else 32))
        blocks = rng.choice(["4,8,16,32", "2,4,8,16", "8,16", "16", "32", "8"] if n_req <= 32 else ["2,4,8,16", "8"])
        ctx_hi = _log_int(rng, 64, min(8192, 200000 // n_req))
        c = {"op": op, "model": model, "n_req": n_req, "blocks": blocks, "ctx_lo": rng.randrange(0, ctx_hi // 2),
             "ctx_hi": ctx_hi, "branches": rng.choice([0, 0, 1, 2]) if n_req <= 8 else 0, "batch": batch}
        if op == "round":
            c.update(logits=rng.choice(["f32", "bf16"]), host=rng.random() < 0.6)
        return c
    if op == "prefill":
        n_req = rng.choice([1, 1, 2, 3, 4])
        chunk_hi = _log_int(rng, 64, 1900 // n_req)
        return {"op": op, "model": rng.choice(["8b", "8b", "small"]), "n_req": n_req, "chunk_lo": chunk_hi // 2 + 1,
                "chunk_hi": chunk_hi, "ctx_lo": 0, "ctx_hi": _log_int(rng, 1, 8192), "batch": batch}
    if op == "device_rounds":
        return {"op": op, "model": "8b", "n_req": _log_int(rng, 1, 16), "rounds": rng.randrange(2, 5),
                "block": rng.choice([8, 16, 32]), "ctx_lo": 100, "ctx_hi": _log_int(rng, 200, 4096), "batch": batch}
    if op == "verify":
        logits = rng.choice(["f32", "bf16"])
        return {"op": op, "n_req": _log_int(rng, 1, 128 if logits == "bf16" else 64), "drafts": rng.randrange(1, 33),
                "block": rng.choice([0, 8, 16, 32]), "vocab": rng.choice([128256, 152064, 32000, 2048, 50257]), "logits": logits, "host": rng.random() < 0.7}
    return {"op": op, "model": "8b", "n_pos": _log_int(rng, 1, 8192), "pos0": rng.choice([0, rng.randrange(0, 2000)])}


# ---- what a program has in hand ---------------------------------------------------------------------------------------
def _descriptor(case):
    if case["op"] == "prefill":
        rng = np.random.default_rng(case["batch"])
        n = case["n_req"]
        chunk = rng.integers(case["chunk_lo"], case["chunk_hi"] + 1, size=n)
        ctx = np.linspace(case["ctx_lo"], case["ctx_hi"], n).astype(int) if n > 1 else [case["ctx_hi"]]
        return synth.fixed_descriptor(ctx, chunk, [0] * n, seed=case["batch"])
    if case["op"] == "device_rounds":
        rng = np.random.default_rng(case["batch"])
        n = case["n_req"]
        ctx = rng.integers(case["ctx_lo"], case["ctx_hi"] + 1, size=n)
        room = case["rounds"] * 33 + 64           # what the rounds append at most
        d = synth.fixed_descriptor(ctx, [1] * n, [room] * n, seed=case["batch"])
        d.block_size = np.full(n, case["block"], dtype=np.int32)
        return d
    blocks = [int(b) for b in case["blocks"].split(",")]
    d = synth.batch_descriptor(case["n_req"], blocks, None, case["ctx_lo"], case["ctx_hi"], seed=case["batch"])
    return synth.with_correction_branches(d, _shape(case).vocab, case["branches"], seed=case["batch"]) if case["branches"] else d


def _successor(t, vocab):
    return (5 * t + 7) % vocab                    # a permutation: 5 divides none of the vocabulary sizes


# brings the successor's logit to about 13 (10 for the small models), against a spread of about 1.3 among the others; the
# share of the token's embedding in the last hidden state falls with the width of the layers
_LEAD = {"tiny": 10.0, "small": 10.0, "8b": 25.0, "14b": 33.0}


def _weights(name, seed):
    shape = _shape({"model": name})
    W = synth.model_weights(shape, seed=seed, device="cuda")
    depth = 1.0 / math.sqrt(2.0 * shape.n_layers)
    for t in W["wo"] + W["w_down"]:
        t.mul_(depth)
    W["embed"].mul_(50.0)
    lead = _LEAD[name] / shape.hidden
    for i in range(0, shape.vocab, 16384):
        ids = torch.arange(i, min(i + 16384, shape.vocab), device="cuda")
        W["lm_head"][_successor(ids, shape.vocab)] += W["embed"][ids] * lead
    return W


def _drafts(desc, vocab, seed):
    """Verify tokens per request: y_0, then drafts that the verifier accepts each with probability 3/4."""
    rng = np.random.default_rng(seed)
    ys = []
    for v in desc.verify_len:
        y = [int(rng.integers(0, vocab - 1))]
        while len(y) < v:
            y.append(_successor(y[-1], vocab) if rng.random() < 0.75 else int(rng.integers(0, vocab - 1)))
        ys.append(y[:v])
    return ys


def _pool(ctx, n_pages, seed):
    """A pool whose committed positions hold K and V of unit variance."""
    pool = torch.empty(ctx.kv_pool_bytes(n_pages) // 2, dtype=torch.bfloat16, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    for i in range(0, pool.numel(), 1 << 28):
        pool[i:i + (1 << 28)].normal_(generator=g)
    return pool


def _capacity(rows):
    n = 32
    while n < rows:
        n *= 2
    return n


# what hangs on the second candidate is left out where whole forwards produce the logits: behind the successor the
# candidates are near ties of random weights (`verify` returns these outputs)
_SKIP = ("top2", "p2", "risky_n", "risky_index", "risky_token")


def _verify_out(batch, host, skip=()):
    out = binding.VerifyOut(batch.n_req, batch.n_tok, batch.n_ver, host=host)
    for name in skip:
        setattr(out.c, name, None)
    return out


def prepare(case, seed):
    op = case["op"]
    if op == "verify":
        n, v, b = case["n_req"], case["drafts"] + 1, case["block"]
        rows = n * (v + b)
        dtype = torch.bfloat16 if case["logits"] == "bf16" else torch.float32
        logits = synth.logits_normal(rows, case["vocab"], seed=seed, device="cuda", dtype=dtype)
        top = torch.cat([logits[i:i + 1024].argmax(dim=1) for i in range(0, rows, 1024)]).cpu().numpy()
        accept = synth.planted_accept_lengths(n, v - 1, seed=seed)
        y = synth.plant_drafts(top.reshape(n, v + b)[:, :v], n, v - 1, accept, case["vocab"], seed=seed).reshape(-1)
        shape = synth.ModelShape(n_layers=0, hidden=64, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=64,
                                 vocab=-(-case["vocab"] // 16) * 16)
        if shape.vocab != case["vocab"]:          # rows of an odd vocabulary come padded with -inf, as engines hand them over
            padded = torch.full((rows, shape.vocab), -math.inf, dtype=dtype, device="cuda")
            padded[:, :case["vocab"]] = logits
            logits = padded
        ctx = binding.Context(binding.make_config(shape, n, rows, 1))
        batch = binding.Batch([0] * n, [v] * n, [b] * n, y)
        return {"op": op, "ctx": ctx, "batch": batch, "logits": logits, "out": _verify_out(batch, case["host"])}
    shape = _shape(case)
    if op in ("kv_write", "kv_read"):
        n_pos, pos0 = case["n_pos"], case["pos0"]
        pt, n_pages = synth.page_tables([pos0], [n_pos], PAGE, seed=seed, spare_pages=16)
        ctx = binding.Context(binding.make_config(shape, 1, 32, pt.shape[1]))
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        s = {"op": op, "ctx": ctx, "layers": shape.n_layers, "pt": pt[0], "n_pages": n_pages, "pos0": pos0, "n_pos": n_pos}
        if op == "kv_write":
            s["pool"] = binding.alloc_kv_pool(ctx, n_pages)
            kv = torch.empty((2, shape.n_layers, n_pos, shape.n_kv_heads, shape.head_dim), dtype=torch.bfloat16, device="cuda")
            s["k"], s["v"] = kv.normal_(generator=g)
        else:
            s["pool"] = _pool(ctx, n_pages, seed)
        return s
    desc = _descriptor(case)
    max_pages = desc.page_table.shape[1]
    if op == "attention":
        ctx = binding.Context(binding.make_config(shape, desc.n_req, _capacity(desc.n_tokens), max_pages))
        pool = _pool(ctx, desc.n_pages, seed)
        batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, None, desc.page_table, pool, desc.n_pages,
                              **desc.branch_kwargs())
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        q = torch.empty((shape.n_layers, desc.n_tokens, shape.n_q_heads, shape.head_dim), dtype=torch.bfloat16, device="cuda")
        q.normal_(generator=g)
        return {"op": op, "ctx": ctx, "pool": pool, "batch": batch, "q": q, "o": torch.empty_like(q)}
    W = _weights(case["model"], seed)
    ys = _drafts(desc, shape.vocab, seed)
    if op == "device_rounds":
        # (every round may carry a reused block of up to 32 verify tokens and draft another one)
        cfg = binding.make_config(shape, desc.n_req, desc.n_req * 64, max_pages)
        ctx = binding.Context(cfg, W)
        pool = _pool(ctx, desc.n_pages, seed)
        dev = binding.DeviceBatch(desc.ctx_len, desc.verify_len, desc.block_size, ys, 32, desc.page_table, pool, desc.n_pages,
                                  rows_hint=desc.n_req * 2 * case["block"])
        log = binding.RoundLog(desc.n_req, case["rounds"], case["rounds"] * 33)
        # the rule with one certainty bin: its choice depends on the last block and on whether it was accepted
        table = synth.policy_table(n_bins=1)
        ctx.recg_policy_load(table["blocks"], table["s_edges"], table["value"], table["cost"])
        z = lambda dt: torch.zeros(desc.n_req, dtype=dt, device="cuda")
        state = {"e1": z(torch.float32), "e2": z(torch.float32), "block_index": z(torch.int32), "full": z(torch.int32)}
        planted = torch.as_tensor(synth.acceptance_chain_lengths(case["rounds"], desc.n_req, seed=case["batch"]), device="cuda")
        first = [t.clone() for t in (dev.ctx_len, dev.verify_len, dev.block_size, dev.verify_tokens)]
        return {"op": op, "ctx": ctx, "pool": pool, "dev": dev, "log": log, "policy": state, "planted": planted,
                "next_block": z(torch.int32), "first": first, "rounds": case["rounds"], "weights": W}
    flags = binding.FLAG_LOGITS_BF16 if case.get("logits") == "bf16" else 0
    ctx = binding.Context(binding.make_config(shape, desc.n_req, _capacity(desc.n_tokens), max_pages, flags), W)
    pool = _pool(ctx, desc.n_pages, seed)
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, [t for y in ys for t in y], desc.page_table, pool,
                          desc.n_pages, **desc.branch_kwargs())
    s = {"op": op, "ctx": ctx, "pool": pool, "batch": batch, "weights": W}
    if op == "round":
        s["out"] = _verify_out(batch, case["host"], _SKIP)
    return s


# ---- one pass -----------------------------------------------------------------------------------------------------------
def _logits(ctx, lg):
    t = binding.device_view(lg.data, (lg.n_rows, lg.vocab), torch.bfloat16 if lg.dtype == binding.DTYPE_BF16 else torch.float32)
    t.owner = ctx          # the memory is the context's: the view keeps it alive
    return t


def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "round":
        lg = ctx.recg_step(s["batch"])
        got = ctx.recg_verify(s["batch"], out=s["out"])
        return {"logits": _logits(ctx, lg), **{k: got[k] for k in got if k not in _SKIP}}
    if op == "prefill":
        # the step leaves the chunk's K/V in the pool; its logits are what sampling goes on from
        return {"logits": _logits(ctx, ctx.recg_step(s["batch"]))}
    if op == "verify":
        return ctx.recg_verify(s["batch"], s["logits"], out=s["out"])
    if op == "attention":
        for layer in range(s["q"].shape[0]):
            ctx.recg_attention(s["batch"] if layer == 0 else None, layer, s["q"][layer], s["o"][layer])
        return s["o"]
    if op == "kv_write":
        for layer in range(s["layers"]):
            ctx.recg_kv_write(s["pool"], s["n_pages"], layer, s["pt"], s["pos0"], s["k"][layer], s["v"][layer])
        return s["pool"]
    if op == "kv_read":
        return [ctx.recg_kv_read(s["pool"], s["n_pages"], layer, s["pt"], s["pos0"], s["n_pos"]) for layer in range(s["layers"])]
    # device_rounds: the batch starts at its first round, then nothing waits for the host
    dev, log, policy = s["dev"], s["log"], s["policy"]
    for t, t0 in zip((dev.ctx_len, dev.verify_len, dev.block_size, dev.verify_tokens), s["first"]):
        t.copy_(t0)
    for t in (log.n_tokens, log.tokens, policy["e1"], policy["e2"], policy["block_index"], policy["full"]):
        t.zero_()
    for r in range(s["rounds"]):
        ctx.recg_step_device(dev)
        ctx.recg_verify_device()
        ctx.recg_policy_step(policy, s["next_block"])
        ctx.recg_next_round(dev, r, s["next_block"], s["planted"][r], log)
    return {"tokens": log.tokens, "n_tokens": log.n_tokens, "accept_len": log.accept_len, "block_size": log.block_size,
            "verify_len": log.verify_len, "entropy_mean": log.entropy_mean, "ctx_len": dev.ctx_len,
            "verify_tokens": dev.verify_tokens, "e1": policy["e1"]}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------------
def _forward_work(shape, ctx_len, verify_len, draft_rows, rows, logits_bytes, weights=True):
    """Weights, the K/V of every request and the logits once; every multiplication that Eq. 1's mask lets through."""
    H, d, nq, nkv, nl = shape.hidden, shape.head_dim, shape.n_q_heads, shape.n_kv_heads, shape.n_layers
    T = float(np.sum(rows))
    kv_tokens = float(np.sum(ctx_len) + T)
    v = np.asarray(verify_len, dtype=np.float64)
    seen = float(np.sum(v * np.asarray(ctx_len) + v * (v + 1) / 2 + np.asarray(draft_rows) * (np.asarray(ctx_len) + rows)))
    b = nl * kv_tokens * nkv * d * 4.0
    f = nl * 4.0 * d * nq * seen
    if weights:
        params = nl * ((nq + 2 * nkv) * d * H + nq * d * H + 3.0 * shape.ffn * H) + shape.vocab * H
        b += 2.0 * params + T * shape.vocab * logits_bytes
        f += 2.0 * T * params
    else:
        b += nl * 4.0 * T * nq * d        # q in, o out
    return {"bytes": b, "flops": f}


def work(case):
    op = case["op"]
    if op == "verify":
        n = case["n_req"] * (case["drafts"] + 1.0 + case["block"]) * case["vocab"]
        return {"bytes": n * (2 if case["logits"] == "bf16" else 4), "flops": 5.0 * n}
    shape = _shape(case)
    if op in ("kv_write", "kv_read"):
        return {"bytes": 8.0 * shape.n_layers * case["n_pos"] * shape.n_kv_heads * shape.head_dim, "flops": 0.0}
    d = _descriptor(case)
    if op == "device_rounds":
        # every round streams the weights; its rows follow from the planted lengths, taken here as one block verified and
        # one drafted in every second round
        rows = np.full(case["n_req"], 1 + case["block"])
        w = _forward_work(shape, d.ctx_len, rows * 0 + 1, rows - 1, rows, 4)
        return {k: case["rounds"] * x for k, x in w.items()}
    return _forward_work(shape, d.ctx_len, d.verify_len, d.rows - d.verify_len, d.rows,
                         2 if case.get("logits") == "bf16" else 4, weights=op != "attention")


def tolerance(case):
    """What another correct implementation shows at the same precision: about four times the distance between the tcgen05
    kernels and the mma.sync kernels (other tiles, other order of every sum).  Measured for whole forwards: logits 6e-3 to
    9e-3 (2-norm), 4e-2 at the worst element, no integer; for attention 2.4e-3 and 1e-2."""
    op = case["op"]
    if op in ("kv_write", "kv_read"):
        return "exact"
    if op == "verify":
        return {"rel": 1e-5, "max": 1e-4}          # fp32 sums; integers as they are
    if op == "attention":
        return {"rel": 1e-2, "max": 5e-2}
    return {"rel": 2.5e-2, "max": 0.15}
