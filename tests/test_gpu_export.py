"""dmc_cache_export_heads and its padded form (GPU).

Heads of 1 to 300 slots into buffers one below, at and one above a block's 64
slots and the longest head, with ids that repeat and ids that do not exist. Both
forms copy the same slots (checked against each other and against a buffer large
enough for all); the plain one leaves the other rows as they were, the padded
one sets them to zero.
"""
import pytest
import torch

import paper_2403_09636_gb300 as P
from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("cap", [1, 63, 64, 65, 300, 321])
def test_padded_and_plain_export(cuda_dev, cap, dtype, D):
    wl = S.Workload("export", 1, 3, 4, 4, D, dtype, (1, 300), 0, ("choice", (1.0, 3.0)), 0.5, seed=77)
    cache = H.cache_for(wl, cuda_dev)
    pr = S.gen_prompt(wl, 0, cuda_dev)
    cache.prefill(0, pr["q0"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"])
    ids = [0, 11, 5, 5, -1, 12, 7]
    want = cache.export_heads(0, ids, 400)
    lens = cache.lengths(0).flatten().tolist()
    assert want[3].tolist() == [lens[i] if 0 <= i < 12 else -1 for i in ids]
    dt = wl.torch_dtype
    t_ids = torch.tensor(ids, dtype=torch.int32, device=cuda_dev)
    for call, rest in ((P.dmc_cache_export_heads, 7.0), (P.dmc_cache_export_heads_padded, 0.0)):
        k = torch.full((len(ids), cap, D), 7.0, dtype=dt, device=cuda_dev)
        v, z = k.clone(), torch.full((len(ids), cap), 7.0, device=cuda_dev)
        ln = torch.zeros(len(ids), dtype=torch.int32, device=cuda_dev)
        s = torch.cuda.current_stream().cuda_stream
        assert call(cache.handle, 0, len(ids), t_ids.data_ptr(), cap, k.data_ptr(), v.data_ptr(), z.data_ptr(),
                    ln.data_ptr(), s) == P.DMC_OK
        assert torch.equal(ln, want[3])
        for i, n in enumerate(ln.tolist()):
            m = min(max(n, 0), cap)
            for got, w in ((k, want[0]), (v, want[1]), (z, want[2])):
                assert torch.equal(got[i, :m], w[i, :m])
                assert bool((got[i, m:] == rest).all())
    assert bool((want[0][:, 301:] == 0).all())
