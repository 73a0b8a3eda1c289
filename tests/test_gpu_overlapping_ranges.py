"""Single-layer decode calls between launches over several layers (GPU).

Steps alternate between decode(1) and a launch over layers 0 and 1, whose ranges share
a layer, with every token a slot of its own over page boundaries. Slots and counts have
to be those of one launch per layer, bit for bit; so have the outputs of the tensor-core
kernel, and those of the other within its tolerance (its split follows the grid).
"""
import pytest
import torch

from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,dtype", [(8, "bf16"), (2, "bf16"), (1, "bf16"), (1, "f32")])
def test_ranges_that_share_a_layer(cuda_dev, group, dtype):
    wl = S.Workload(f"ranges_{group}_{dtype}", 2, 4, 8 * group, 8, 128, dtype, (20, 700), 48, ("fixed", 1.0), 0.5, seed=41)
    prompts = [S.gen_prompt(wl, layer, cuda_dev) for layer in range(2)]
    steps = [[S.gen_decode(wl, layer, t, cuda_dev) for layer in range(2)] for t in range(wl.decode_steps)]
    results = []
    for walk in (False, True):
        cache = H.cache_for(wl, cuda_dev)
        for layer, p in enumerate(prompts):
            cache.prefill(layer, p["q0"], p["k"], p["v"], p["cu_seqlens"], p["max_seqlen"])
        q, k, v = (torch.stack([torch.stack([x[layer][n] for layer in range(2)]) for x in steps]) for n in "qkv")
        out = torch.zeros_like(q)
        extra = torch.zeros_like(q[:, 0])
        torch.cuda.synchronize()
        for t in range(0, wl.decode_steps, 2):
            cache.decode(1, q[t, 1], k[t, 1], v[t, 1], extra[t])  # layer 1 has a token more per pair of steps
            if walk:
                cache.decode_layers(0, q[t + 1], k[t + 1], v[t + 1], out[t + 1])
            else:
                torch.cuda.synchronize()
                for layer in range(2):
                    cache.decode(layer, q[t + 1, layer], k[t + 1, layer], v[t + 1, layer], out[t + 1, layer])
                    torch.cuda.synchronize()
        assert cache.status()[:2] == (0, 0)
        lens = [cache.lengths(layer) for layer in range(2)]
        heads = [cache.export_heads(layer, list(range(32)), 760) for layer in range(2)]
        results.append((out, extra, lens, heads))
    (o0, e0, l0, h0), (o1, e1, l1, h1) = results
    for a, b in zip(l0, l1):
        assert torch.equal(a, b)
    for x, y in zip(h0, h1):
        for a, b in zip(x, y):
            assert torch.equal(a, b)
    for a, b in ((o0, o1), (e0, e1)):
        if group > 1:
            assert torch.equal(a, b)
        else:
            assert float((a.float() - b.float()).abs().max()) <= H.TOL[dtype]
