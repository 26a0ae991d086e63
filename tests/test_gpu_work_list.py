"""The attention work list where its segments change: causal chunks around the 32-token tiles, their pairs and the 64-token
KV blocks (early tiles of a chunk read fewer blocks than late ones), and more requests and segments than the list's CTA has
threads."""
import numpy as np
import pytest
import torch

from oracle import recg_oracle as orc
from paper_2609_34388_b200 import binding, synth
from tests._util import f64, oracle_cfg, oracle_weights
from tests.test_gpu_ops import ATTN_TOL, run_attention_case
from tests.test_gpu_step import HID_TOL, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [0, 5, 130])
@pytest.mark.parametrize("v,b", [(31, 0), (32, 0), (33, 0), (64, 0), (65, 0), (96, 1), (257, 0), (120, 40)])
def test_causal_chunks(L, v, b):
    for shape in (synth.llama8b_shape(1), synth.tiny_shape()):
        assert run_attention_case(shape, [(L, v, b), (77, 40, 0), (3, 1, 2)], seed=v + L) < ATTN_TOL


def test_more_requests_than_threads():
    shape = synth.ModelShape(n_layers=1, hidden=64, n_q_heads=4, n_kv_heads=2, head_dim=128, ffn=64, vocab=64)
    reqs = [(i % 19, 1 + i % 3, i % 2) for i in range(1100)] + [(40, 70, 0), (500, 33, 0)]
    assert run_attention_case(shape, reqs, seed=3) < ATTN_TOL


@pytest.mark.parametrize("reqs", [[(0, 1, 0)], [(200, 8, 8)], [(300, 16, 16)], [(340, 16, 16)], [(100, 40, 0), (250, 33, 10)],
                                  [(64, 100, 0)], [(400, 60, 4)] * 3, [(300, 8, 8)] * 18, [(300, 8, 8)] * 19])
def test_whole_tiles_of_short_contexts(reqs):
    """On both sides of the rule that leaves tiles uncut: about six blocks of context, and as many tiles as CTAs."""
    for shape in (synth.llama8b_shape(1), synth.tiny_shape()):
        assert run_attention_case(shape, reqs, seed=len(reqs) + reqs[0][0]) < ATTN_TOL


@pytest.mark.parametrize("n_req", [2, 257, 300, 513])
def test_tokens_of_many_requests(n_req):
    """A whole step finds every row's request among more requests than the embedding kernel's CTA has threads (256), some of
    one row, some that only draft: the rows of the first and last request and of those around the 256th and 512th."""
    shape = synth.ModelShape(n_layers=1, hidden=128, n_q_heads=2, n_kv_heads=1, head_dim=64, ffn=256, vocab=512)
    W = synth.model_weights(shape, seed=0, dtype=torch.bfloat16)
    v = [0 if r % 7 == 3 else 1 + r % 2 for r in range(n_req)]
    b = [2 if v[r] == 0 or r % 3 == 0 else 0 for r in range(n_req)]
    L = [r % 5 for r in range(n_req)]
    desc = synth.fixed_descriptor(L, v, b, seed=9)
    ctx = binding.Context(binding.make_config(shape, n_req, desc.n_tokens, desc.page_table.shape[1]), to_dev(W))
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    checked = [r for r in (0, 1, 254, 255, 256, 257, 258, 511, 512, n_req - 1) if r < n_req]
    kvs, ys = {}, []
    for r in range(n_req):
        ys.append(synth.token_ids(v[r], shape.vocab, seed=r + 1).tolist() if v[r] else [])
        K, V = synth.kv_values(max(L[r], 1), 1, 64, seed=r)
        kvs[r] = (K[:L[r]], V[:L[r]])
        if L[r]:
            ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[r], 0, kvs[r][0].cuda(), kvs[r][1].cuda())
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, [t for y in ys for t in y], desc.page_table, pool, desc.n_pages)
    logits = f64(ctx.logits_tensor(ctx.recg_step(batch)))
    ctx.recg_sync()
    first = np.concatenate([[0], np.cumsum(np.array(v) + np.array(b))])
    for r in checked:
        K, V = kvs[r]
        ref, _, _ = orc.fused_round_cached(oracle_cfg(shape), oracle_weights(W), [(K.double().numpy(), V.double().numpy())], L[r], ys[r], b[r])
        got = logits[first[r]:first[r + 1]]
        assert np.max(np.abs(got - ref)) <= HID_TOL * np.max(np.abs(ref)), r
    ctx.recg_free()


@pytest.mark.parametrize("n_layers", [1, 3])
def test_attention_right_behind_a_verification_with_pages(n_layers):
    """A verification of given logits lays its batch out, and the attention calls that follow name no batch: they work on that
    layout, also the first one, in front of which no kernel of any size has run (device results: nothing waits for the host).
    Batches of few and many requests take turns, so that a list of the batch before would show."""
    shape = synth.ModelShape(n_layers=n_layers, hidden=512, n_q_heads=4, n_kv_heads=2, head_dim=128, ffn=64, vocab=64)
    sets = [[(300, 3, 2)], [(40, 1, 3), (700, 2, 0), (5, 4, 4)], [(20 * i % 333, 1 + i % 3, i % 2) for i in range(40)]]
    descs = [synth.fixed_descriptor([r[0] for r in s], [r[1] for r in s], [r[2] for r in s], seed=9 + i) for i, s in enumerate(sets)]
    n_pages = max(d.n_pages for d in descs)
    ctx = binding.Context(binding.make_config(shape, 40, max(d.n_tokens for d in descs), max(d.page_table.shape[1] for d in descs)))
    pool = binding.alloc_kv_pool(ctx, n_pages, fill="normal")
    work = []
    for i, d in enumerate(descs):
        y = synth.token_ids(int(d.verify_len.sum()), shape.vocab, seed=i)
        batch = binding.Batch(d.ctx_len, d.verify_len, d.block_size, y, d.page_table, pool, n_pages)
        logits = synth.logits_normal(d.n_tokens, shape.vocab, seed=i, device="cuda")
        q = synth.queries(d.n_tokens * n_layers, 4, 128, seed=i).cuda().view(n_layers, d.n_tokens, 4, 128)
        want = torch.empty_like(q)
        for l in range(n_layers):
            ctx.recg_attention(batch, l, q[l], want[l])
        ctx.recg_sync()
        work.append((batch, logits, q, want, binding.VerifyOut(d.n_req, d.n_tokens, len(y), host=False)))
    got = []
    for rep in range(60):
        batch, logits, q, want, out = work[rep % 3]
        o = torch.full_like(q, float("nan"))
        torch.cuda.synchronize()
        ctx.recg_verify(batch, logits, out=out)
        for l in range(n_layers):
            ctx.recg_attention(None, l, q[l], o[l])
        got.append(o)
    ctx.recg_sync()
    for rep, o in enumerate(got):
        assert torch.equal(o, work[rep % 3][3]), rep
    ctx.recg_free()
