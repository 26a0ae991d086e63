"""K/V import and export at the edges of their launches: remainders of a CTA's chunks, pages entered in the middle, and more
pages than one launch carries page ids for."""
import pytest
import torch

from paper_2609_34388_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,n_kv", [(64, 2), (128, 1), (128, 8), (128, 5)])
@pytest.mark.parametrize("pos0,n_pos", [(0, 1), (5, 16), (15, 2), (37, 403), (3, 4093), (3, 4094), (3, 14333), (3, 14334), (9, 14400)])
def test_kv_round_trip_touches_its_positions_only(head_dim, n_kv, pos0, n_pos):
    shape = synth.ModelShape(n_layers=2, hidden=64, n_q_heads=n_kv, n_kv_heads=n_kv, head_dim=head_dim, ffn=64, vocab=64)
    if (n_kv * 3 * head_dim) % 128:
        pytest.skip("the context asks for a qkv width of whole 128 columns")
    pt, n_pages = synth.page_tables([pos0], [n_pos], 16, seed=n_pos, spare_pages=3)
    ctx = binding.Context(binding.make_config(shape, 1, 32, pt.shape[1]))
    pool = binding.alloc_kv_pool(ctx, n_pages)
    k, v = synth.kv_values(n_pos, n_kv, head_dim, seed=n_pos + 1, device="cuda")
    k[k == 0] = 1.0
    v[v == 0] = 1.0
    ctx.recg_kv_write(pool, n_pages, 1, pt[0], pos0, k, v)
    assert int(torch.count_nonzero(pool)) == 2 * n_pos * n_kv * head_dim          # nothing else was written
    assert int(torch.count_nonzero(pool[:pool.numel() // 2])) == 0                # ... and nothing in the other layer
    kb, vb = ctx.recg_kv_read(pool, n_pages, 1, pt[0], pos0, n_pos)
    assert torch.equal(kb, k) and torch.equal(vb, v)
    for i in {0, n_pos // 2, n_pos - 1}:                                          # every position where a read alone looks for it
        kb, vb = ctx.recg_kv_read(pool, n_pages, 1, pt[0], pos0 + i, 1)
        assert torch.equal(kb[0], k[i]) and torch.equal(vb[0], v[i])
    # the K and V rows of a page lie inside the tiles of the page its table names
    tiles = pool.view(2, n_pages, n_kv, 2, 16 * head_dim)[1]
    i = n_pos // 2
    page = int(pt[0][(pos0 + i) // 16])
    for h in range(n_kv):
        assert set(k[i, h].tolist()) <= set(tiles[page, h, 0].tolist())
        assert set(v[i, h].tolist()) <= set(tiles[page, h, 1].tolist())
    ctx.recg_sync()
    ctx.recg_free()
