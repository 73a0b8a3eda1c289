"""Prompt attention with inputs that are not numbers (GPU).

A token attends over slots and tokens up to itself, so a later token whose query,
key or value is NaN or infinite must not change an earlier token's output. A query
tile of 128 rows (128 / G tokens) shares its probabilities' product with V, where a
hidden slot's zero weight times NaN is NaN, so what is promised is a tile's grain:
the outputs of every tile before the token's are the same bits as without it. (Two
tiles share a work item and its K/V tiles.) And a NaN importance neuron of a token
that opens a slot must not lose the opening: every later token sees that slot, so
every later output of its KV head is NaN.
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


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("cr", [1.0, 3.0])
@pytest.mark.parametrize("G", [1, 2, 4, 8])
def test_a_later_tile_does_not_reach_an_earlier_one(cuda_dev, G, cr, bad):
    """n tokens: seven tiles and a few rows; the tokens made bad are the first, one
    inside and the last of a tile, for the tiles of one item and of the next."""
    TT = 128 // G
    n = 7 * TT + 5
    wl = _wl(f"later_g{G}_{cr}", 1, 3 * G, 3, (n, n), ("fixed", cr), seed=1000 + G)
    pr = S.gen_prompt(wl, 0, cuda_dev, full_q=True)
    clean, lens = _run(wl, pr)
    assert bool(torch.isfinite(clean).all())
    for tile in (1, 2, 3, 5, 7):
        for t in sorted({tile * TT, min(tile * TT + TT // 2 + 1, n - 1), min(tile * TT + TT, n) - 1}):
            d = {x: pr[x].clone() if x in "qkv" else pr[x] for x in pr}
            for x in "qkv":
                d[x][t, :, 1:] = bad
            out, got = _run(wl, d)
            assert torch.equal(got, lens)
            assert torch.equal(out[:tile * TT], clean[:tile * TT]), (tile, t)


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
