"""Prompt attention at the edges of its tiles (GPU).

A work item is 256 query rows (256 / G tokens) of one head, as two tiles of 128;
slots come in tiles of 128 read as pages of 32, the prompt's rows as 128-token
chunks. Prompts one below, at and one above those sizes, with every token a slot
of its own (so the slot count hits the same edges), are checked against the fp64
oracle (outputs and slots, 2e-2 as for every bf16 cache). The arena starts as
NaNs, so that anything read beyond what was written shows. A second test puts
NaNs into the next sequence of the packed prompt, whose rows lie in the same
tiles: the first sequence's outputs have to stay as they were, bit for bit.
"""
import pytest
import torch

from paper_2403_09636_gb300 import synthetic as S
from tests.test_gpu_prefill_attention import _cache, _check_layer, _wl

pytestmark = pytest.mark.gpu

LENGTHS = [1, 31, 63, 65, 127, 128, 129, 255, 256, 257, 384, 400]


def _nan_arena(cache):
    cache.arena.fill_(0xFF)
    cache.reset()


@pytest.mark.parametrize("G", [1, 2, 4, 8])
@pytest.mark.parametrize("n", LENGTHS)
def test_edges_of_tiles_match_the_oracle(cuda_dev, G, n):
    for cr in (1.0, 3.0):
        wl = _wl(f"edge_g{G}_{n}", 2, 2 * G, 2, (n, n), ("fixed", cr), seed=600 + n)
        cache = _cache(wl)
        _nan_arena(cache)
        pr = S.gen_prompt(wl, 0, cuda_dev, full_q=True)
        out = torch.full_like(pr["q"], float("nan"))
        cache.prefill_attention(0, pr["q"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"], out)
        assert cache.status()[:2] == (0, 0)
        bad = _check_layer(wl, cache, 0, pr, out)
        assert not bad, (cr, bad[:8])


@pytest.mark.parametrize("G", [1, 8])
@pytest.mark.parametrize("n", [1, 33, 100, 130, 250, 300])
def test_the_next_sequence_does_not_reach_into_a_tile(cuda_dev, G, n):
    wl = _wl(f"next_g{G}_{n}", 2, 2 * G, 2, (n, n), ("fixed", 2.0), seed=700 + n)
    pr = S.gen_prompt(wl, 0, cuda_dev, full_q=True)
    outs = []
    for dirty in (False, True):
        if dirty:
            for t in ("q", "k", "v"):
                pr[t][n:, :, 1:] = float("nan")
        cache = _cache(wl)
        _nan_arena(cache)
        out = torch.empty_like(pr["q"])
        cache.prefill_attention(0, pr["q"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"], out)
        assert cache.status()[:2] == (0, 0)
        outs.append(out[:n].clone())
    assert bool(torch.isfinite(outs[0]).all())
    assert torch.equal(outs[0], outs[1])
