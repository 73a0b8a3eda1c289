"""Precision of the weights in grouped-query decoding (GPU).

The tensor-core kernel multiplies the softmax weights with V in bf16, as a rounded value
and what the rounding left (16 bits or more together), so an output is off by its own
rounding to bf16 and little else: it has to be the bf16 of the fp64 attention over the
cache's slots but where that lies next to a rounding boundary. A weight is off by at
most 2^-17, a sum of weighted values by about as much of its largest terms, an output's
bf16 spacing is 2^-7 of it at most: with outputs some times smaller than their terms
that is a boundary crossed in well under 2 % of them. With weights rounded to bf16 once
(2^-9) it is in tens of percent.
"""
import math

import pytest
import torch

from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [0, 12])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,Hkv,G,n", [(1, 2, 8, 3000), (4, 8, 2, 500), (16, 8, 8, 70), (3, 4, 5, 900)])
def test_outputs_are_the_rounded_attention(cuda_dev, B, Hkv, G, n, D, window):
    wl = S.Workload(f"precise_{B}_{Hkv}_{G}_{D}", 1, B, Hkv * G, Hkv, D, "bf16", (n, n), 1, ("fixed", 2.0), 0.5,
                    seed=300 + n, q_scale=2.0)
    cache = H.cache_for(wl, cuda_dev, window=window)
    p, x = S.gen_prompt(wl, 0, cuda_dev), S.gen_decode(wl, 0, 0, cuda_dev)
    cache.prefill(0, p["q0"], p["k"], p["v"], p["cu_seqlens"], p["max_seqlen"])
    out = torch.empty_like(x["q"])
    cache.decode(0, x["q"], x["k"], x["v"], out)
    K, V, _, ln = cache.export_heads(0, list(range(B * Hkv)), n + 1)
    assert cache.status()[:2] == (0, 0)
    q = x["q"].double().view(B * Hkv, G, D).clone()
    q[..., 0] = 0.0
    s = torch.einsum("hgd,hnd->hgn", q, K.double()) / math.sqrt(D)
    s = s.masked_fill(torch.arange(n + 1, device=cuda_dev) >= ln[:, None, None], -math.inf)
    ref = torch.einsum("hgn,hnd->hgd", torch.softmax(s, 2), V.double()).to(torch.bfloat16)
    wrong = (out.view(B * Hkv, G, D) != ref).double().mean().item()
    assert wrong <= 0.02, wrong
