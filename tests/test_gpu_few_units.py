"""Decode layers with fewer page units than worker warps, or about as many (GPU).

Both decode kernels then run fewer workers than the grid has warps. Checked
against the fp64 oracle at the edges: one head of one slot, heads cut into one
part per page, and a cache whose unit count crosses the grid's warp count while
it is decoded (64 heads of 18 pages are 1,216 units, of 19 pages 1,280; a GB300
runs 1,216 warps of the CUDA-core kernel over one layer, 1,520 over several). The tolerance is the
dtype's (slots stored in bf16 round at every merge: 2e-2; fp32: 1e-4).
"""
import pytest

from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


def _wl(name, B, Hq, Hkv, D, dtype, prompt, steps, cr, seed):
    return S.Workload(name, 2, B, Hq, Hkv, D, dtype, prompt, steps, ("fixed", cr), 1.0 if dtype == "f32" else 0.5,
                      seed=seed)


CASES = [
    _wl("one_head_one_slot", 1, 1, 1, 128, "bf16", (1, 1), 5, 1.0, 71),
    _wl("one_head_f32", 1, 1, 1, 64, "f32", (33, 33), 40, 1.0, 72),
    _wl("mha_b1_long", 1, 4, 4, 128, "bf16", (4000, 4000), 6, 1.0, 73),
    _wl("mha_crosses_the_warp_count", 8, 8, 8, 128, "bf16", (572, 572), 10, 1.0, 74),
    _wl("mha_crosses_the_walk_s_warp_count", 10, 8, 8, 128, "bf16", (572, 572), 10, 1.0, 81),
    _wl("f32_virtual_heads_b1", 1, 6, 2, 128, "f32", (700, 700), 6, 2.0, 75),
    _wl("gqa8_b1_one_slot", 1, 8, 1, 128, "bf16", (1, 1), 5, 1.0, 76),
    _wl("gqa8_b1_long", 1, 16, 2, 128, "bf16", (6000, 6000), 6, 1.0, 77),
    _wl("gqa2_d64_b1", 1, 4, 2, 64, "bf16", (3000, 3000), 6, 1.5, 78),
    _wl("gqa5_b4", 4, 20, 4, 128, "bf16", (500, 1500), 8, 2.0, 79),
    _wl("gqa8_crosses_the_warp_count", 9, 16, 2, 64, "bf16", (1050, 1060), 12, 1.0, 80),
]


@pytest.mark.parametrize("launch", ["stream", "layers"])
@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_few_units_match_the_oracle(cuda_dev, wl, launch):
    run = H.Run(wl, cuda_dev, H.all_samples(wl), launch=launch)
    assert run.len_ok, run.len_msgs[:5]
    bad = run.compare()
    assert not bad, bad[:10]


@pytest.mark.parametrize("launch", ["stream", "layers"])
def test_many_grouped_heads(cuda_dev, launch):
    """4,800 KV heads: the unit prefixes take the shared memory of the tensor-core
    kernel's third tile per warp."""
    wl = _wl("gqa2_many_heads", 600, 16, 8, 128, "bf16", (1, 70), 3, 2.0, 82)
    run = H.Run(wl, cuda_dev, H.random_samples(wl, 64, seed=5), launch=launch)
    assert run.len_ok, run.len_msgs[:5]
    bad = run.compare()
    assert not bad, bad[:10]
