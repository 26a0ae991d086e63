"""The per-request end of verification where its paths change: requests on both sides of the rows it keeps in shared memory
(256), accept scans that cross a warp's 32 rows, few and many vocabulary chunks per row, results on the host and on the device."""
import math

import numpy as np
import pytest
import torch

from oracle import recg_oracle as orc
from paper_2609_34388_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("host", [True, False])
@pytest.mark.parametrize("reqs,vocab", [
    # (verify rows, accepted drafts, mask rows)
    ([(5, 2, 0)], 128256),                                   # 32 vocabulary chunks per row
    ([(33, 31, 2), (34, 32, 1), (1, 0, 40)], 32000),
    ([(255, 254, 1), (256, 100, 0), (1, 0, 0)], 2048),       # 256 rows: kept in shared memory
    ([(256, 255, 1), (0, 0, 257), (300, 64, 33)], 2048),     # more rows than that
    ([(9, 8, 8)] * 700, 2048),                               # one chunk per row
])
def test_rows_of_a_request(reqs, vocab, host):
    v, acc, b = (np.array(x, dtype=np.int32) for x in zip(*reqs))
    T = int((v + b).sum())
    shape = synth.ModelShape(n_layers=0, hidden=64, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=64, vocab=vocab)
    ctx = binding.Context(binding.make_config(shape, len(reqs), T, 1))
    logits = synth.logits_normal(T, vocab, seed=T, dtype=torch.float32)
    top = logits.numpy().argmax(axis=1)                      # fp32 draws of this size have no equal maxima
    rng = np.random.default_rng(T)
    y, t0 = [], 0
    for r in range(len(reqs)):
        if v[r]:
            yr = rng.integers(0, vocab, size=v[r])
            yr[1:acc[r] + 1] = top[t0:t0 + acc[r]]
            if acc[r] + 1 < v[r]:
                yr[acc[r] + 1] = (top[t0 + acc[r]] + 1) % vocab
            y += yr.tolist()
        t0 += v[r] + b[r]
    batch = binding.Batch(np.zeros(len(reqs)), v, b, y)
    got = ctx.recg_verify(batch, logits.cuda(), host=host)
    ctx.recg_sync()
    if not host:
        got = {k: t.cpu().numpy() for k, t in got.items()}
    t0 = tv0 = tb0 = 0
    for r in range(len(reqs)):
        n = v[r] + b[r]
        ref = orc.verify_round(logits[t0:t0 + n].double().numpy(), y[tv0:tv0 + v[r]], int(b[r]))
        st = ref["stats"]
        assert int(got["accept_len"][r]) == ref["accept_len"] == acc[r]
        assert int(got["n_emitted"][r]) == ref["n_emitted"] and int(got["cont_hit"][r]) == int(ref["cont_hit"])
        assert int(got["new_ctx_len"][r]) == ref["n_emitted"]
        assert got["emitted"][tv0:tv0 + v[r]].tolist() == ref["emitted"] + [-1] * (v[r] - ref["n_emitted"])
        assert got["next_draft"][tb0:tb0 + b[r]].tolist() == ref["next_draft"]
        assert got["top1"][t0:t0 + n].tolist() == [s["top1"] for s in st]
        assert got["top2"][t0:t0 + n].tolist() == [s["top2"] for s in st]
        # fp32 sums of up to 128256 terms and the hardware's 2^x (2 ulp): 1e-5 relative
        np.testing.assert_allclose(got["p1"][t0:t0 + n], [s["p1"] for s in st], rtol=1e-5)
        np.testing.assert_allclose(got["p2"][t0:t0 + n], [s["p2"] for s in st], rtol=1e-5)
        np.testing.assert_allclose(got["entropy"][t0:t0 + n], [s["entropy"] for s in st], rtol=1e-5)
        assert abs(float(got["entropy_mean"][r]) - ref["entropy_mean"]) <= 2e-5 * max(1.0, ref["entropy_mean"])
        # every draft of such logits is risky (margins below 0.5): the count, the earliest two and their second candidates
        rows = max(int(b[r]) - 1, 0)
        assert got["risky_n"][3 * r:3 * r + 3].tolist() == [rows, 0, 0]
        want = [1 + i if i < rows else -1 for i in range(2)]
        assert got["risky_index"][6 * r:6 * r + 6].tolist() == want + [-1] * 4
        assert got["risky_token"][6 * r:6 * r + 6].tolist() == [st[v[r] + i]["top2"] if i > 0 else -1 for i in want] + [-1] * 4
        assert got["slot_state"][t0:t0 + n].tolist() == [0] * n          # no page table: no slots
        assert int(got["freed_pages"][r]) == 0 and (got["freed_page_ids"][t0:t0 + n] == -1).all()
        t0 += n
        tv0 += v[r]
        tb0 += b[r]
    ctx.recg_free()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab", [3, 255, 257, 1023, 1025, 1279, 2049, 5001, 50257])
def test_rows_of_any_alignment(vocab, dtype):
    """Rows of an odd vocabulary begin on every element boundary: most have no 16-byte vectors, and the elements of a thread end in
    every remainder of four.  Every second row has many equal values: the lowest index wins."""
    logits = synth.logits_normal(9, vocab, seed=vocab, device="cuda", dtype=dtype)
    logits[::2] = logits[::2].round()
    got = binding.recg_row_stats_static(logits)
    torch.cuda.synchronize()
    host = logits.double().cpu().numpy()
    for r in range(9):
        want = orc.row_stats(host[r])
        assert int(got["top1"][r]) == want["top1"] and int(got["top2"][r]) == want["top2"], r
        for k in ("p1", "p2", "entropy"):          # as above: fp32 sums, 2^x of the hardware
            assert abs(float(got[k][r]) - want[k]) <= 1e-5 * max(want[k], 1e-3 if k == "entropy" else 0.0), (k, r)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("mask", ["lowest", -1e30, -2e9, -1e9, -math.inf])
@pytest.mark.parametrize("vocab", [2048, 50257, 128256])
def test_masked_logits(vocab, mask, dtype):
    """Masked entries carry no probability whatever value stands for them, also where a thread or a whole chunk of the vocabulary
    sees nothing else: a masked tail (a padded vocabulary), a masked head, all but every 97th and all but three entries."""
    value = torch.finfo(dtype).min if mask == "lowest" else mask
    logits = synth.logits_normal(4, vocab, seed=vocab, device="cuda", dtype=dtype)
    keep = torch.zeros((4, vocab), dtype=torch.bool, device="cuda")
    keep[0, :vocab - vocab // 3] = True
    keep[1, vocab // 2:] = True
    keep[2, ::97] = True
    keep[3, [5, vocab // 2, vocab - 1]] = True
    logits = logits.masked_fill(~keep, value)
    got = binding.recg_row_stats_static(logits)
    torch.cuda.synchronize()
    host, kept = logits.double().cpu().numpy(), keep.cpu().numpy()
    for r in range(4):
        ids = np.nonzero(kept[r])[0]
        want = orc.row_stats(host[r][ids])       # the entries that are not masked are all there is
        assert int(got["top1"][r]) == ids[want["top1"]] and int(got["top2"][r]) == ids[want["top2"]], r
        for k in ("p1", "p2", "entropy"):
            assert abs(float(got[k][r]) - want[k]) <= 1e-5 * max(want[k], 1e-3 if k == "entropy" else 0.0), (k, r)
