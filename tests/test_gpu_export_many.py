"""Exports whose heads are cut into more pieces than a plain export has blocks (GPU).

A plain export (dmc_cache_export_heads) spreads a bounded number of blocks over its
heads, each taking every n-th piece of 64 slots; with many heads a block walks several
pieces. Both forms, with one below, exactly and more heads than blocks, a capacity far
above the heads' lengths, and ids that repeat, against one head exported at a time.
"""
import pytest
import torch

import paper_2403_09636_gb300 as P
from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 500, 1215, 1216, 1300])
def test_blocks_walk_the_pieces_of_a_head(cuda_dev, n):
    D, cap = 64, 450
    wl = S.Workload("export_many", 1, 2, 4, 4, D, "bf16", (150, 440), 0, ("fixed", 1.0), 0.5, seed=78)
    cache = H.cache_for(wl, cuda_dev, max_slots=4096, num_pages=400)
    pr = S.gen_prompt(wl, 0, cuda_dev)
    cache.prefill(0, pr["q0"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"])
    one = [cache.export_heads(0, [h], cap) for h in range(8)]
    ids = torch.arange(n, dtype=torch.int32, device=cuda_dev) % 8
    s = torch.cuda.current_stream().cuda_stream
    for call, rest in ((P.dmc_cache_export_heads, 7.0), (P.dmc_cache_export_heads_padded, 0.0)):
        k = torch.full((n, cap, D), 7.0, dtype=torch.bfloat16, device=cuda_dev)
        v, z = k.clone(), torch.full((n, cap), 7.0, device=cuda_dev)
        ln = torch.zeros(n, dtype=torch.int32, device=cuda_dev)
        assert call(cache.handle, 0, n, ids.data_ptr(), cap, k.data_ptr(), v.data_ptr(), z.data_ptr(),
                    ln.data_ptr(), s) == P.DMC_OK
        for h in range(min(n, 8)):
            m = int(one[h][3][0])
            for got, want in ((k, one[h][0]), (v, one[h][1]), (z, one[h][2])):
                assert bool((got[h::8, :m] == want[:, :m]).all())
                assert bool((got[h::8, m:] == rest).all())
            assert bool((ln[h::8] == m).all())
    assert cache.status()[:2] == (0, 0)
