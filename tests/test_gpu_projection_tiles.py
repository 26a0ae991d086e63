"""Projections where their tiles change: token tiles of every width (multiples of 16, and of 32 for CTA pairs), one and several
of them, rows in the last chunk of 32, feature tiles that the matrix does not fill, every way of cutting K, and the epilogues
of a whole step at such sizes."""
import numpy as np
import pytest
import torch

from oracle import recg_oracle as orc
from paper_2609_34388_b200 import binding, synth
from tests._util import f64, oracle_cfg, oracle_weights
from tests.test_gpu_step import HID_TOL, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,sk", [(0, 0), (64, 0), (64, 1), (128, 1), (128, 2), (256, 0), (256, 1), (256, 2), (384, 0), (384, 1),
                                     (512, 0), (512, 1), (512, 2)])
@pytest.mark.parametrize("N,K", [(16, 64), (144, 320), (1040, 1024), (2304, 512)])
def test_rows_around_the_tiles(tile, sk, N, K):
    shape = synth.tiny_shape()
    ctx = binding.Context(binding.make_config(shape, 1, 8, 1))
    ctx.recg_debug_gemm_config(tile, sk)
    g = torch.Generator().manual_seed(N + K)
    w = (torch.randn((N, K), generator=g) * 0.05).to(torch.bfloat16)
    xs = torch.randn((700, K), generator=g).to(torch.bfloat16)
    ref = xs.double().numpy() @ w.double().numpy().T
    wd, xd = w.cuda(), xs.cuda()
    for M in (1, 15, 16, 17, 31, 33, 47, 64, 65, 112, 129, 160, 176, 208, 240, 255, 256, 257, 272, 300, 511, 513, 700):
        for dt in (torch.float32, torch.bfloat16):
            buf = torch.full((M + 2, N), float("nan"), dtype=dt, device="cuda")       # two guard rows behind the matrix
            ctx._check(binding.lib().recg_linear(ctx.h, xd.data_ptr(), wd.data_ptr(), buf.data_ptr(), M, N, K,
                                                 binding.DTYPE_F32 if dt == torch.float32 else binding.DTYPE_BF16))
            ctx.recg_sync()
            got = f64(buf)
            assert np.isnan(got[M:]).all(), (M, str(dt))
            # fp32 sums of K <= 1024 exact bf16 products: sqrt(K) 2^-24 < 1e-5 of the largest; bf16 output: half an ulp, 2^-9
            tol = 1e-5 if dt == torch.float32 else 2.0 ** -8
            assert np.max(np.abs(got[:M] - ref[:M])) <= tol * np.max(np.abs(ref)), (M, str(dt))
    ctx.recg_free()


@pytest.mark.parametrize("flags", [0, binding.FLAG_SIMT_GEMM])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_results_of_any_alignment(dt, flags):
    """A result that starts 0 to 16 bytes behind a 16-byte boundary: computed where a kernel can store it (bf16: multiples of 8
    bytes; fp32: any element, multiples of 16 bytes with the mma.sync kernel), an error anywhere else; x and w likewise."""
    M, N, K = 37, 144, 320
    ctx = binding.Context(binding.make_config(synth.tiny_shape(), 1, 8, 1, flags))
    g = torch.Generator().manual_seed(1)
    w = (torch.randn((N, K), generator=g) * 0.05).to(torch.bfloat16)
    x = torch.randn((M, K), generator=g).to(torch.bfloat16)
    ref = x.double().numpy() @ w.double().numpy().T
    wd, xd = w.cuda(), x.cuda()
    size = 4 if dt == torch.float32 else 2
    need = 8 if dt == torch.bfloat16 else (16 if flags else 4)
    call = lambda xp, wp, yp: binding.lib().recg_linear(ctx.h, xp, wp, yp, M, N, K, binding.DTYPE_F32 if size == 4 else binding.DTYPE_BF16)
    for off in range(0, 17, size):
        buf = torch.full((M * N + 32,), float("nan"), dtype=dt, device="cuda")
        i = off // size
        assert buf.data_ptr() % 16 == 0
        status = call(xd.data_ptr(), wd.data_ptr(), buf.data_ptr() + off)
        assert status == (0 if off % need == 0 else 1), off
        ctx.recg_sync()
        got = f64(buf)
        assert np.isnan(got[:i]).all() and np.isnan(got[i + M * N:]).all(), off
        if status:
            assert np.isnan(got).all()
        else:          # the bounds of the test above
            tol = 1e-5 if size == 4 else 2.0 ** -8
            assert np.max(np.abs(got[i:i + M * N].reshape(M, N) - ref)) <= tol * np.max(np.abs(ref)), off
    y = torch.empty((M, N), dtype=dt, device="cuda")
    assert call(xd.data_ptr() + 8, wd.data_ptr(), y.data_ptr()) == 1 and call(xd.data_ptr(), wd.data_ptr() + 2, y.data_ptr()) == 1
    ctx.recg_sync()
    ctx.recg_free()


@pytest.mark.parametrize("force", [(0, 0), (64, 1), (256, 2), (384, 0), (512, 1)])
@pytest.mark.parametrize("head_dim,n_q,n_kv", [(64, 2, 1), (128, 1, 1), (64, 6, 2)])
def test_step_of_a_model_that_fills_no_tile(head_dim, n_q, n_kv, force):
    """hidden, FFN and vocabulary are not multiples of a feature tile; 1 to 380 rows."""
    shape = synth.ModelShape(n_layers=2, hidden=192, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=head_dim, ffn=320, vocab=2064)
    W = synth.model_weights(shape, seed=0, dtype=torch.bfloat16)
    synth.perturb_norm_gains(W)
    ocfg, W64 = oracle_cfg(shape), oracle_weights(W)
    Wd = to_dev(W)
    for specs in ([(0, 1, 0)], [(5, 3, 30)], [(40, 100, 29), (0, 0, 1)], [(33, 250, 0), (7, 8, 8), (100, 60, 54)]):
        L, v, b = (list(t) for t in zip(*specs))
        desc = synth.fixed_descriptor(L, v, b, seed=9)
        ctx = binding.Context(binding.make_config(shape, len(specs), desc.n_tokens, desc.page_table.shape[1]), Wd)
        ctx.recg_debug_gemm_config(*force)
        pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
        pool.fill_(float("nan"))
        ys, kvs = [], []
        for r in range(len(specs)):
            kv = []
            for l in range(shape.n_layers):
                K, V = synth.kv_values(max(L[r], 1), n_kv, head_dim, seed=100 * r + l)
                K, V = K[:L[r]], V[:L[r]]
                if L[r]:
                    ctx.recg_kv_write(pool, desc.n_pages, l, desc.page_table[r], 0, K.cuda(), V.cuda())
                kv.append((K.double().numpy(), V.double().numpy()))
            kvs.append(kv)
            ys.append(synth.token_ids(v[r], shape.vocab, seed=r + 1).tolist() if v[r] else [])
        batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, [t for y in ys for t in y], desc.page_table, pool,
                              desc.n_pages)
        logits = f64(ctx.logits_tensor(ctx.recg_step(batch)))
        ctx.recg_sync()
        hidden = f64(ctx.recg_debug_buffer(0))
        t0 = 0
        for r in range(len(specs)):
            n = v[r] + b[r]
            ref, ref_kv, ref_h = orc.fused_round_cached(ocfg, W64, kvs[r], L[r], ys[r], b[r])
            assert np.max(np.abs(logits[t0:t0 + n] - ref)) <= HID_TOL * np.max(np.abs(ref)), (specs, r)
            assert np.max(np.abs(hidden[t0:t0 + n] - ref_h)) <= HID_TOL * np.max(np.abs(ref_h)), (specs, r)
            for l, (K, V) in enumerate(ref_kv):
                kg, vg = ctx.recg_kv_read(pool, desc.n_pages, l, desc.page_table[r], L[r], n)
                assert np.max(np.abs(f64(kg) - K[L[r]:])) <= HID_TOL * np.max(np.abs(K[L[r]:])), (specs, r, l)
                assert np.max(np.abs(f64(vg) - V[L[r]:])) <= HID_TOL * np.max(np.abs(V[L[r]:])), (specs, r, l)
            t0 += n
        ctx.recg_free()


@pytest.mark.parametrize("M,N,K", [(333, 19088, 2048), (376, 9600, 4096), (700, 14336, 4096), (701, 19088, 2048)])
def test_ragged_end_cut_in_narrower_tiles(M, N, K):
    """Sizes at which the columns of the last wave are cut over K, in token tiles narrower than the others' (one to seven such
    columns, two to eight parts per tile, the last feature tile half empty)."""
    ctx = binding.Context(binding.make_config(synth.tiny_shape(), 1, 8, 1))
    g = torch.Generator().manual_seed(M)
    w = (torch.randn((N, K), generator=g) * 0.05).to(torch.bfloat16).cuda()
    x = torch.randn((M, K), generator=g).to(torch.bfloat16).cuda()
    ref = f64(x.double() @ w.double().T)
    for rep in range(2):
        got = f64(ctx.recg_linear(x, w))
        # fp32 sums of 4096 exact bf16 products: sqrt(K) 2^-24 = 4e-6 of the largest
        assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref)), rep
    ctx.recg_free()


@pytest.mark.parametrize("M,N,K", [(333, 19088, 2048), (376, 9600, 4096), (700, 14336, 4096), (701, 19088, 2048), (333, 28672, 2048),
                                   (376, 28672, 2048)])
def test_sizes_of_the_ragged_end_tests_are_cut(M, N, K):
    """The sizes of the tests above and below are divided as those say: some of the columns cut, in narrower token tiles."""
    ctx = binding.Context(binding.make_config(synth.tiny_shape(), 1, 8, 1))
    p = ctx.recg_debug_gemm_plan(M, N, K)
    assert 0 < p["cut_columns"] < p["columns"] and p["cut_width"] < p["width"] and not p["cluster"], p
    assert p["cut_range"] < p["cut_columns"] * K // 64           # several teams, so tiles in several parts
    ctx.recg_free()


@pytest.mark.parametrize("n", [333, 376])
def test_ragged_end_cut_of_a_whole_step(n):
    """The same division inside a step: 28672 gate and up rows of 2048 at these row counts (SwiGLU epilogue, RMSNorm folded)."""
    shape = synth.ModelShape(n_layers=1, hidden=2048, n_q_heads=4, n_kv_heads=1, head_dim=128, ffn=14336, vocab=2064)
    W = synth.model_weights(shape, seed=0, dtype=torch.bfloat16)
    ctx = binding.Context(binding.make_config(shape, 1, n, 64), to_dev(W))
    desc = synth.fixed_descriptor([0], [n], [0], seed=9)
    pool = binding.alloc_kv_pool(ctx, desc.n_pages, fill=None)
    pool.fill_(float("nan"))
    y = synth.token_ids(n, shape.vocab, seed=1).tolist()
    batch = binding.Batch(desc.ctx_len, desc.verify_len, desc.block_size, y, desc.page_table, pool, desc.n_pages)
    logits = f64(ctx.logits_tensor(ctx.recg_step(batch)))
    ctx.recg_sync()
    none = (np.zeros((0, 1, 128)), np.zeros((0, 1, 128)))
    ref, _, _ = orc.fused_round_cached(oracle_cfg(shape), oracle_weights(W), [none], 0, y, 0)
    assert np.max(np.abs(logits - ref)) <= HID_TOL * np.max(np.abs(ref))
    ctx.recg_free()
