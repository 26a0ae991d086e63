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
from tests.test_gpu_overlap import run_attention_case as run_branch_case
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


def work_list(ctx_len, rows, verify_len, n_kv, tok_per_tile=32, n_ctas=148):
    """The attention work list's rule, restated: (request, first tile, number of tiles, KV range in tokens) of every item.  Two
    neighbouring row tiles make a pair with a line of CTA pairs of its own; a segment costs its 64-token blocks and six (a pair) or
    four more, and the owners of a line share its sum evenly.  (Not for batches whose tiles are left whole.)"""
    tiles = [-(-n // tok_per_tile) for n in rows]
    assert n_kv * sum(tiles) > n_ctas

    def segments(pair):
        for r, rt in enumerate(tiles):
            for i in [i for _ in range(n_kv) for i in (range(0, rt - 1, 2) if pair else range(rt - 1, rt) if rt % 2 else ())]:
                last = min(rows[r], (i + (2 if pair else 1)) * tok_per_tile)
                yield r, i, -(-(ctx_len[r] + (last if last <= verify_len[r] else rows[r])) // 64)
    wa, wb = (sum(nb + (6 if pair else 4) for _, _, nb in segments(pair)) for pair in (True, False))
    pairs = min(max(int(0.5 * n_ctas * 2 * wa / (2 * wa + wb) + 0.5), 1), n_ctas // 2) if wa else 0
    if wb and n_ctas - 2 * pairs < 1:
        pairs = (n_ctas - 1) // 2
    items = []
    for pair, owners, work, extra in ((True, pairs, wa, 6), (False, n_ctas - 2 * pairs, wb, 4)):
        at, per = 0, -(-work // owners) if owners and work else 1
        for r, i, nb in segments(pair):
            g0 = at + extra
            at = g0 + nb
            for c in range(g0 // per, (at - 1) // per + 1):
                items.append((r, i, 2 if pair else 1, 64 * (max(g0, c * per) - g0), 64 * (min(at, (c + 1) * per) - g0)))
    return items


def stages_done_again(scores, first, end):
    """Per softmax group of an item: the stages in which a row of `scores` (in powers of two) outgrows its reference by 2^8."""
    out = []
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
    n_kv, n_req, v, b = 8, 20, 2, 2
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
    items = work_list(lens, [v + b] * n_req, [v] * n_req, n_kv)
    kvs, again = [], []
    for r, L in enumerate(lens):
        n = L + v + b
        pos = torch.arange(n)
        step = (pos == 1200 + 40 * r).float() if profile == "late" else (pos // 128 + (pos % 64 == 5)).float()
        masked = (pos < n // 3) if low else torch.zeros(n, dtype=torch.bool)
        k = torch.zeros((n, n_kv, 128))
        k[:, :, 0] = (masked * low / 2.0 ** 20)[:, None]
        k[:, :, 1] = (~masked * (base / side if base else 0.0))[:, None]
        k[:, :, 2] = (~masked * 28.0 * step)[:, None]      # a step is a factor of 2^28.6
        k = k.to(torch.bfloat16)
        _, vals = synth.kv_values(n, n_kv, 128, seed=r)
        vals = 0.25 * vals.float() + 1.0 - 2.0 * (step % 2)[:, None, None]
        if profile == "late":              # what has been summed before the step still weighs as much as the step's token
            vals[step == 0] *= 2.0 ** 18
        vals = vals.to(torch.bfloat16)
        kvs.append((k, vals))
        ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[r], 0, k.cuda(), vals.cuda())
        scores = (f64(q[0, 0]) @ f64(k[:, 0]).T) / (np.sqrt(128.0) * np.log(2.0))
        again += [a for i in items if i[0] == r for a in stages_done_again(scores, i[3], i[4])]
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
        # (P and the result are rounded to bf16, 2^-9 each; heads with and without steps have results of different size)
        for heads in (slice(0, None, 2), slice(1, None, 2)):
            assert np.max(np.abs(got[rows, heads] - ref[:, heads])) <= ATTN_TOL * np.max(np.abs(ref[:, heads])), r
    ctx.recg_free()


def test_rows_that_see_nothing_of_their_first_stages():
    """Correction branches behind long verify chunks: a branch row sees the context up to its position and its own block, nothing
    of the hundreds of tokens between, and items begin there.  Its reference maximum is then set in a later stage of the item."""
    shape = synth.llama8b_shape(1)
    reqs = [(70 + 55 * i, 330 + 37 * i, 32, [(1 + i, 0)], 20 + i) for i in range(10)]
    rows = [v + b + 1 + bc for _, v, b, _, bc in reqs]
    late = [set(), set()]
    for r, tile, n_tiles, first, end in work_list([q[0] for q in reqs], rows, [q[1] for q in reqs], 8):
        L, v, b, corr, bc = reqs[r]
        _, vis, _ = orc.overlap_round_rows(L, v, b, corr, bc)
        seen = np.asarray(vis)[32 * tile:32 * (tile + n_tiles), :end]
        for g in (0, 64):
            stages = np.array([seen[:, t:t + 64].any(axis=1) for t in range(first + g, end, 128)]).reshape(-1, seen.shape[0])
            if len(stages):
                late[g // 64] |= set(np.argmax(stages, axis=0)[stages.any(axis=0)].tolist())
    assert all(max(s) >= 2 for s in late), late        # (in both softmax groups)
    assert run_branch_case(shape, reqs, seed=61) < ATTN_TOL


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
    """Inside a step a warp keeps a row: 1 to 18 tiles with up to 141 parts (18 at a time), and 27."""
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


@pytest.mark.parametrize("d", [64, 128])
def test_step_loses_no_part(d):
    """One row tile in 141 parts, inside a step.  The attention's result stands out in the logits (embeddings scaled down), and every
    64 tokens of the context have values of their own: one part less would be seen."""
    L, v, b = 9000, 6, 2
    shape = synth.ModelShape(n_layers=1, hidden=128, n_q_heads=2, n_kv_heads=1, head_dim=d, ffn=128, vocab=256)
    W = synth.model_weights(shape, seed=0, dtype=torch.bfloat16)
    W["embed"] = W["embed"] * 2.0 ** -8
    desc = synth.fixed_descriptor([L], [v], [b], seed=3)
    ctx = binding.Context(binding.make_config(shape, 1, desc.n_tokens, desc.page_table.shape[1]), to_dev(W))
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    K, V = synth.kv_values(L, 1, d, seed=4)
    V = torch.sign(V[::64].float()).repeat_interleave(64, dim=0)[:L].to(torch.bfloat16)
    ctx.recg_kv_write(pool, desc.n_pages, 0, desc.page_table[0], 0, K.cuda(), V.cuda())
    y = synth.token_ids(v, shape.vocab, seed=1).tolist()
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, y, desc.page_table, pool, desc.n_pages)
    got = f64(ctx.logits_tensor(ctx.recg_step(batch)))
    ctx.recg_sync()

    def oracle(without):
        vis = orc.fused_round_visibility(L, v, b).copy()
        vis[:, without] = False
        ids = y + [oracle_cfg(shape).mask_id()] * b
        return orc.decoder_rows(oracle_cfg(shape), oracle_weights(W), ids, np.arange(L, L + v + b), vis, [(f64(K), f64(V))], None)[0]
    ref = oracle(slice(0, 0))
    tol = HID_TOL * np.max(np.abs(ref))
    for part in (0, 17, 18, 31, 32, 100, 139):
        assert np.max(np.abs(oracle(slice(64 * part, 64 * part + 64)) - ref)) > 3 * tol, part
    assert np.max(np.abs(got - ref)) <= tol
    ctx.recg_free()
