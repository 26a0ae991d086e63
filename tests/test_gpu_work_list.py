"""The attention work list where its segments change: causal chunks around the 32-token tiles, their pairs and the 64-token
KV blocks (early tiles of a chunk read fewer blocks than late ones), and more requests and segments than the list's CTA has
threads."""
import pytest

from paper_2609_34388_b200 import synth
from tests.test_gpu_ops import ATTN_TOL, run_attention_case

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
