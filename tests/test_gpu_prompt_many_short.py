"""Prompt attention over many short prompts (GPU).

With more work items than SMs a CTA takes several, and those with rows for one query
tile only take the two tiles' places in turn. Prompts of 1 to 3 query tiles, whole and
continued, in one call, against the same sequences in calls of so few that every CTA
has one item: the same bits, slots and counts.
"""
import pytest
import torch

from paper_2403_09636_gb300 import DmcCache

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 2, 4, 8])
@pytest.mark.parametrize("longest", [20, 128, 300])
def test_many_items_per_cta(cuda_dev, G, longest):
    B, H, D, few = 240, 2, 128, 10
    longest = max(longest // G, 3)
    g = torch.Generator(device=cuda_dev).manual_seed(G * longest)
    results = []
    parts = []
    for part in range(2):
        lens = torch.randint(0, longest + 1, (B,), generator=g, device=cuda_dev)
        cu = torch.cat([torch.zeros(1, dtype=torch.int64, device=cuda_dev), lens.cumsum(0)]).int()
        n = int(cu[-1])
        q, k, v = (torch.randn((n, heads, D), generator=g, device=cuda_dev).bfloat16() for heads in (H * G, H, H))
        parts.append((q, k, v, cu))
    for step in (B, few):
        cache = DmcCache(1, B, H * G, H, D, torch.bfloat16, 2 * longest + 1, B * H * (longest // 16 + 2),
                         max(p[1].shape[0] for p in parts))
        cache.arena.fill_(0xFF)  # what was never written is NaN
        cache.reset()
        outs = []
        for q, k, v, cu in parts:
            out = torch.full_like(q, float("nan"))
            for s in range(0, B, step):
                lo, hi = int(cu[s]), int(cu[s + step])
                if hi > lo:
                    cache.prefill_attention(0, q[lo:hi], k[lo:hi], v[lo:hi], cu[s:s + step + 1] - lo, longest,
                                            out[lo:hi], first_seq=s)
            outs.append(out)
        assert cache.status()[:2] == (0, 0)
        heads = cache.export_heads(0, list(range(B * H)), 2 * longest + 1)
        results.append(outs + list(heads))
    assert all(bool(torch.isfinite(x).all()) for x in results[0][:2])
    for a, b in zip(*results):
        assert torch.equal(a, b)
