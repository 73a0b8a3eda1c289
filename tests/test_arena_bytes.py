"""What a cache's arena holds for prompts (CPU).

The prompt's decisions and first slot indexes take 20 bytes per 128-token chunk and KV
head. The carried sums and omegas of prompt attention come on top only in the caches it
serves: bf16, head_dim 128, 1, 2, 4 or 8 query heads per KV head, no window.
"""
import pytest

import paper_2403_09636_gb300 as P
from paper_2403_09636_gb300 import build as B

CHUNKS, HEADS = 1000, 4


def _prompt_bytes(dtype=P.DMC_BF16, head_dim=128, group=1, window=0):
    def need(tokens):
        return P.dmc_cache_required_bytes(P.dmc_cache_config(1, 2, HEADS * group, HEADS, head_dim, dtype, 32, 100, 50,
                                                             tokens, window))
    return need(CHUNKS * 128) - need(0)


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()


@pytest.mark.parametrize("kw", [dict(dtype=P.DMC_F32), dict(head_dim=64), dict(window=1), dict(group=3),
                                dict(group=16)])
def test_caches_without_prompt_attention_hold_decisions_only(kw):
    assert _prompt_bytes(**kw) == pytest.approx(CHUNKS * HEADS * 20, abs=1024)


@pytest.mark.parametrize("group", [1, 2, 4, 8])
def test_caches_with_prompt_attention_hold_its_sums(group):
    per_chunk = 20 + (2 * 128 + 1) * 4 + 128 * 4
    assert _prompt_bytes(group=group) == pytest.approx(CHUNKS * HEADS * per_chunk, abs=2048)
