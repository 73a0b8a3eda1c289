"""Inconsistent cu_seqlens do not write outside what the heads were given (GPU).

Sequences whose bounds are valid by themselves but overlap share entries of the
prompt's chunk table, so a block may find another sequence's slot index and decisions
there. The fault bit is set, and every write has to stay inside pages that the pool has
handed out: the rest of the pool, filled beforehand, keeps its bytes. (The page-table
rows that nothing allocated hold the same filling, a page id far outside the pool.)
"""
import pytest
import torch

from paper_2403_09636_gb300 import DMC_FAULT_BAD_SEQLENS, DmcCache

pytestmark = pytest.mark.gpu

CUS = [[0, 1000, 200, 1200], [0, 700, 128, 1200], [0, 1000, 640, 700], [600, 1200, 0, 900]]


@pytest.mark.parametrize("cu", CUS)
@pytest.mark.parametrize("kind", ["exact", "window", "attention"])
@pytest.mark.parametrize("append", [0.05, 0.6, 1.0])
def test_overlapping_sequences_stay_inside_their_pages(cuda_dev, kind, cu, append):
    B, H, D, n = len(cu) - 1, 3, 128, 1200
    g = torch.Generator(device=cuda_dev).manual_seed(7)
    q, k, v = (torch.randn((n, H, D), generator=g, device=cuda_dev).bfloat16() for _ in range(3))
    opens = torch.rand((n, H), generator=g, device=cuda_dev) < append
    k[..., 0] = torch.where(opens, -1.0, 1.0).bfloat16()
    pages = B * H * 40 + 64
    c = DmcCache(1, B, H, H, D, torch.bfloat16, 1216, pages, n, window=12 if kind == "window" else 0)
    c.arena.fill_(0xA5)
    c.reset()
    cu_dev = torch.tensor(cu, dtype=torch.int32, device=cuda_dev)
    if kind == "attention":
        c.prefill_attention(0, q, k, v, cu_dev, n, torch.empty_like(q))
    else:
        c.prefill(0, q[..., 0], k, v, cu_dev, n)
    _, bits, used = c.status()
    assert bits == DMC_FAULT_BAD_SEQLENS
    page = 2 * 32 * D * 2
    pool = c.arena[:pages * page].view(pages, page)
    assert used <= pages - 64
    assert bool((pool[used:] == 0xA5).all())
    z = c.arena[pages * page:][:pages * 128].view(pages, 128)  # the pool is a multiple of the arena's alignment
    assert bool((z[used:] == 0xA5).all())
    assert int(c.lengths(0).max()) <= 1200
