"""A cache used from two streams, its calls ordered by events (GPU).

A prompt is compressed into layer 1 on stream B while layer 0 decodes on stream A, and
layer 1 then decodes on B: the decode has to see the whole prompt. The results have to
be, bit for bit, those of the same calls on one stream.
"""
import pytest
import torch

from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,dtype,D", [(1, "bf16", 128), (8, "bf16", 128), (1, "f32", 64)])
def test_a_prompt_of_one_layer_while_another_decodes(cuda_dev, group, dtype, D):
    wl = S.Workload(f"two_{group}_{dtype}", 2, 8, 8 * group, 8, D, dtype, (1500, 2048), 2, ("fixed", 2.0), 0.5, seed=31)
    prompts = [S.gen_prompt(wl, layer, cuda_dev) for layer in range(2)]
    steps = [S.gen_decode(wl, layer, 0, cuda_dev) for layer in range(2)]
    results = []
    for two in (False, True):
        cache = H.cache_for(wl, cuda_dev)
        outs = [torch.zeros_like(x["q"]) for x in steps]
        a = torch.cuda.Stream()
        b = torch.cuda.Stream() if two else a
        torch.cuda.synchronize()

        def prefill(layer, s):
            p = prompts[layer]
            cache.prefill(layer, p["q0"], p["k"], p["v"], p["cu_seqlens"], p["max_seqlen"], stream=s)

        def decode(layer, s):
            x = steps[layer]
            cache.decode(layer, x["q"], x["k"], x["v"], outs[layer], stream=s)

        prefill(0, a)
        b.wait_stream(a)
        prefill(1, b)
        a.wait_stream(b)
        decode(0, a)
        b.wait_stream(a)
        decode(1, b)
        torch.cuda.synchronize()
        assert cache.status()[:2] == (0, 0)
        results.append(outs + [cache.lengths(layer) for layer in range(2)])
    for one, other in zip(*results):
        assert torch.equal(one, other)
