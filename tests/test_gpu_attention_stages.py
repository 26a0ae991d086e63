"""The attention kernel's reference maximum and its combine kernel where their paths change: scores that outgrow the reference in
every stage or never, rows that see nothing of their first stages, and few row tiles (their parts are merged by one, two or four
warps a row)."""
import numpy as np
import pytest
import torch

from oracle import recg_oracle as orc
from paper_2609_34388_b200 import binding, synth
from tests._util import f64, oracle_cfg, oracle_weights
from tests.test_gpu_ops import ATTN_TOL, ops_ctx, run_attention_case
from tests.test_gpu_step import HID_TOL, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["rising", "falling", "steps", "large"])
@pytest.mark.parametrize("L,v,b", [(0, 200, 0), (130, 3, 60), (1000, 16, 16), (2500, 40, 5)])
def test_scores_against_the_standing_reference(kind, L, v, b):
    shape = synth.ModelShape(n_layers=1, hidden=64, n_q_heads=4, n_kv_heads=1, head_dim=128, ffn=64, vocab=64)
    n = L + v + b
    desc = synth.fixed_descriptor([L], [v], [b], seed=L)
    ctx = ops_ctx(shape, 1, desc.n_tokens, desc.page_table.shape[1])
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    q = synth.queries(v + b, 4, 128, seed=5)
    k, vals = synth.kv_values(n, 1, 128, seed=7)
    pos = torch.arange(n, dtype=torch.float32)
    scale = {"rising": 1 + 40 * pos / n, "falling": 41 - 40 * pos / n, "steps": 1 + 12 * (pos // 100 % 4), "large": torch.full((n,), 60.0)}[kind]
    k = (k.float() * scale[:, None, None]).to(torch.bfloat16)
    ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[0], 0, k.cuda(), vals.cuda())
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, None, desc.page_table, pool, desc.n_pages)
    o = torch.full((v + b, 4, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    ctx.recg_attention(batch, 0, q.cuda(), o)
    ctx.recg_sync()
    ref = orc.hybrid_attention(f64(q), f64(k), f64(vals), L, v, b)
    # (the scores reach 300; fp32 sums of 128 exact products of that size are off by less than 300 x 128 x 2^-24 = 2e-3 at worst,
    # 2e-3 of a probability; P and the result are rounded to bf16, 2^-9 each)
    assert np.max(np.abs(f64(o) - ref)) <= ATTN_TOL * np.max(np.abs(ref))
    ctx.recg_free()


def cut_of_single_tiles(kv_len, n_kv, n_ctas=148):
    """The KV ranges [first, end) of every request (per kv head, in tokens) where each request has one row tile: the work list's
    rule, restated (a segment costs its 64-token blocks and four more, and the CTAs share the sum evenly)."""
    blocks = [-(-n // 64) for n in kv_len for _ in range(n_kv)]
    per = -(-sum(n + 4 for n in blocks) // n_ctas)
    cut, at = [], 0
    for n in blocks:
        g0 = at + 4
        at = g0 + n
        ends = [min(g0 + n, (c + 1) * per) - g0 for c in range(g0 // per, (g0 + n - 1) // per + 1)]
        cut.append([(64 * a, 64 * e) for a, e in zip([0] + ends, ends)])
    return cut


def stages_done_again(scores, cut):
    """Stage numbers of every item and softmax group in which a row of `scores` (in powers of two) outgrows its reference."""
    out = []
    for first, end in cut:
        for g in (0, 64):
            ref, again = None, []
            for n, t in enumerate(range(first + g, min(end, len(scores)), 128)):
                top = scores[t:min(t + 64, end)].max()
                if ref is None:
                    ref = top
                elif top > ref + 8:
                    ref = top
                    again.append(n)
            out.append(again)
    return out


@pytest.mark.parametrize("profile,base,low", [("late", 2.0 ** 20, 0), ("late", 2.0 ** 24, 0), ("late", 2.0 ** 26, 0), ("every", 0.0, 0),
                                              ("every", 2.0 ** 24, 0), ("late", 2.0 ** 13, -2.0 ** 40), ("every", 2.0 ** 13, -2.0 ** 40)])
def test_reference_follows_the_scores_exactly(profile, base, low):
    """Scores that outgrow the reference late in an item, or in every stage of it, on top of a common value `base`, and (low) a third
    of the context with scores as of a mask.  Every score is a sum of at most two products and exact in fp32, so nothing but the
    probabilities' and the result's rounding to bf16 stands between the kernel and float64, however large the scores are."""
    n_kv, n_req, v, b = 8, 16, 2, 2
    lens = [1900 + 13 * r for r in range(n_req)]
    shape = synth.ModelShape(n_layers=1, hidden=64, n_q_heads=4 * n_kv, n_kv_heads=n_kv, head_dim=128, ffn=64, vocab=64)
    desc = synth.fixed_descriptor(lens, [v] * n_req, [b] * n_req, seed=1)
    ctx = ops_ctx(shape, n_req, desc.n_tokens, desc.page_table.shape[1])
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    side = 2.0 ** (np.log2(base) // 2) if base else 0.0
    q = torch.zeros((desc.n_tokens, 4 * n_kv, 128))
    q[..., 0], q[..., 1] = 2.0 ** 20, side
    q[:, ::2, 2] = 8.0                   # (every other head sees the steps, the others a plain mean of what is not masked)
    q = q.to(torch.bfloat16)
    cut = cut_of_single_tiles([n + v + b for n in lens], n_kv)
    kvs, again = [], []
    for r, L in enumerate(lens):
        n = L + v + b
        pos = torch.arange(n)
        step = (pos == 1200 + 40 * r).float() if profile == "late" else (pos // 128 + (pos % 64 == 5)).float()
        masked = (pos < n // 3) if low else torch.zeros(n, dtype=torch.bool)
        k = torch.zeros((n, n_kv, 128))
        k[:, :, 0] = (masked * low / 2.0 ** 20)[:, None]
        k[:, :, 1] = (~masked * (base / side if base else 0.0))[:, None]
        k[:, :, 2] = (~masked * 9.0 * step)[:, None]
        k = k.to(torch.bfloat16)
        _, vals = synth.kv_values(n, n_kv, 128, seed=r)
        vals = (0.25 * vals.float() + 1.0 - 2.0 * (step % 2)[:, None, None]).to(torch.bfloat16)
        kvs.append((k, vals))
        ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[r], 0, k.cuda(), vals.cuda())
        scores = (f64(q[0, 0]) @ f64(k[:, 0]).T) / (np.sqrt(128.0) * np.log(2.0))
        again += [a for h in range(n_kv) for a in stages_done_again(scores, cut[r * n_kv + h])]
    # a stage is done again behind the second one, and (steps in every stage) one right behind the other
    assert any(a and a[-1] >= 2 for a in again)
    assert profile == "late" or any(len(a) >= 3 and a[2] == a[0] + 2 for a in again)
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, None, desc.page_table, pool, desc.n_pages)
    o = torch.full((desc.n_tokens, 4 * n_kv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    ctx.recg_attention(batch, 0, q.cuda(), o)
    ctx.recg_sync()
    got = f64(o)
    for r, L in enumerate(lens):
        rows = slice(4 * r, 4 * r + 4)
        ref = orc.hybrid_attention(f64(q[rows]), f64(kvs[r][0]), f64(kvs[r][1]), L, v, b)
        # (P and the result are rounded to bf16, 2^-9 each, against values of at most 2.2)
        assert np.max(np.abs(got[rows] - ref)) <= ATTN_TOL * np.max(np.abs(ref)), r
    ctx.recg_free()


@pytest.mark.parametrize("n_kv,reqs", [
    (8, [(4096, 16, 16)]),                       # 8 tiles: four warps a row
    (8, [(900, 20, 12), (3000, 1, 0)]),          # 16 tiles: two
    (1, [(9000, 30, 2)]),                        # one tile in a part per CTA
    (3, [(1200, 33, 0), (2, 1, 0), (700, 2, 9)]),   # 12 tiles, a pair among them
    (8, [(500, 4, 4), (1500, 8, 8), (2500, 2, 30)]),    # 24 tiles: one warp
])
def test_parts_of_few_tiles(n_kv, reqs):
    for d in (64, 128):
        shape = synth.ModelShape(n_layers=1, hidden=64, n_q_heads=4 * n_kv, n_kv_heads=n_kv, head_dim=d, ffn=64, vocab=64)
        assert run_attention_case(shape, reqs, seed=len(reqs) + n_kv) < ATTN_TOL


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n_kv,reqs", [(1, [(9000, 6, 2)]), (2, [(3000, 30, 10)]), (2, [(700, 1, 3), (2600, 4, 0)]), (9, [(500, 3, 1), (1300, 2, 2)]),
                                       (9, [(500, 3, 1), (1300, 2, 2), (90, 1, 0)])])
def test_step_with_few_tiles(n_kv, reqs, d):
    """Inside a step a warp keeps a row: 1 to 18 tiles with up to 148 parts (18 at a time), and 27."""
    shape = synth.ModelShape(n_layers=1, hidden=128, n_q_heads=2 * n_kv, n_kv_heads=n_kv, head_dim=d, ffn=128, vocab=256)
    W = synth.model_weights(shape, seed=0, dtype=torch.bfloat16)
    L, v, b = ([r[i] for r in reqs] for i in range(3))
    desc = synth.fixed_descriptor(L, v, b, seed=3)
    ctx = binding.Context(binding.make_config(shape, len(reqs), desc.n_tokens, desc.page_table.shape[1]), to_dev(W))
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    kvs, ys = [], []
    for r in range(len(reqs)):
        ys.append(synth.token_ids(v[r], shape.vocab, seed=r + 1).tolist())
        kvs.append(synth.kv_values(L[r], n_kv, d, seed=r))
        ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[r], 0, kvs[r][0].cuda(), kvs[r][1].cuda())
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, [t for y in ys for t in y], desc.page_table, pool, desc.n_pages)
    logits = f64(ctx.logits_tensor(ctx.recg_step(batch)))
    ctx.recg_sync()
    t0 = 0
    for r in range(len(reqs)):
        K, V = kvs[r]
        ref, _, _ = orc.fused_round_cached(oracle_cfg(shape), oracle_weights(W), [(K.double().numpy(), V.double().numpy())], L[r], ys[r], b[r])
        got = logits[t0:t0 + v[r] + b[r]]
        assert np.max(np.abs(got - ref)) <= HID_TOL * np.max(np.abs(ref)), r
        t0 += v[r] + b[r]
    ctx.recg_free()
