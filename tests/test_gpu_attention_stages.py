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
