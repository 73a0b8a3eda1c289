"""Prompt attention with inputs that are not numbers (GPU).

A NaN importance neuron of a token that opens a slot must not lose the opening: every
later token sees that slot, so every later output of its KV head is NaN; the other
heads and the query tiles (128 / G tokens) before the token's stay as they were.
"""
import pytest
import torch

from paper_2403_09636_gb300 import synthetic as S
from tests.test_gpu_prefill_attention import _cache, _wl

pytestmark = pytest.mark.gpu


def _run(wl, pr):
    cache = _cache(wl)
    cache.arena.fill_(0xFF)  # what was never written is NaN
    cache.reset()
    out = torch.empty_like(pr["q"])
    cache.prefill_attention(0, pr["q"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"], out)
    assert cache.status()[:2] == (0, 0)
    return out, cache.lengths(0)


@pytest.mark.parametrize("G", [1, 4])
@pytest.mark.parametrize("sign", [0, 1])
def test_a_nan_importance_keeps_its_opening(cuda_dev, G, sign):
    """Every token opens a slot; one query's gate of one token is a NaN of either sign."""
    n, t, H = 300, 140, 2
    wl = _wl(f"nan_gate_g{G}", 1, H * G, H, (n, n), ("fixed", 1.0), seed=1100 + G)
    pr = S.gen_prompt(wl, 0, cuda_dev, full_q=True)
    clean, lens = _run(wl, pr)
    d = {x: pr[x].clone() if x in "qkv" else pr[x] for x in pr}
    d["q"].view(torch.int16)[t, G, 0] = -1 if sign else 0x7FFF  # KV head 1's first query
    out, got = _run(wl, d)
    assert torch.equal(got, lens)
    assert torch.equal(out[:, :G], clean[:, :G])
    first = t // (128 // G) * (128 // G)  # the tile that holds the token
    assert torch.equal(out[:first, G:], clean[:first, G:])
    assert bool(out[t:, G:].isnan().all())
