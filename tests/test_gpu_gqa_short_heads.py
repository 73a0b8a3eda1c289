"""Grouped queries over short heads (GPU).

A layer of short heads (up to six pages and the new token on average) gives the
tensor-core kernel's workers one unit each. Heads of two to nine units over few and many
KV heads, groups of 2 to 8, both head_dims, one launch per layer and one for both,
against the fp64 oracle (2e-2).
"""
import pytest

from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launch", ["stream", "layers"])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,Hkv,G,prompt", [(1, 8, 2, (40, 40)), (16, 8, 2, (30, 66)), (16, 4, 3, (60, 70)),
                                            (5, 2, 8, (190, 260)), (20, 8, 8, (64, 64))])
def test_short_heads_match_the_oracle(cuda_dev, B, Hkv, G, prompt, D, launch):
    wl = S.Workload(f"short_{B}_{Hkv}_{G}_{D}", 2, B, Hkv * G, Hkv, D, "bf16", prompt, 4, ("fixed", 1.0), 0.5,
                    seed=190 + B + G)
    samples = H.random_samples(wl, min(48, 2 * B * Hkv), seed=7)
    run = H.Run(wl, cuda_dev, samples, launch=launch)
    assert run.len_ok, run.len_msgs[:5]
    bad = run.compare()
    assert not bad, bad[:10]
