"""Decode layers with many heads (GPU).

A cache with more than 3 heads for every 2 warps of the CUDA-core kernel's one-layer
shape (1,824 heads on a GB300, 1,216 warps) takes the shape of launches over several
layers. One below, at and above that line, short heads (a page, a page's edge), every
row width, window grouping and virtual heads, one launch per layer and one for both;
the walk's own warp count (1,824) crossed while decoding; and the static-scratch entry
point, whose partial states follow the shape. Against the fp64 oracle with the
tolerance of the dtype (2e-2 bf16, 1e-4 fp32).
"""
import pytest
import torch

import paper_2403_09636_gb300 as P
from paper_2403_09636_gb300 import synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


def _wl(name, B, Hq, Hkv, D, dtype, prompt, steps, cr, seed):
    return S.Workload(name, 2, B, Hq, Hkv, D, dtype, prompt, steps, ("fixed", cr), 1.0 if dtype == "f32" else 0.5,
                      seed=seed)


CASES = [
    (_wl("heads_1824", 57, 32, 32, 128, "bf16", (20, 40), 3, 1.0, 171), 0),
    (_wl("heads_1825", 73, 25, 25, 128, "bf16", (20, 40), 3, 1.0, 172), 0),
    (_wl("heads_2560", 64, 40, 40, 64, "bf16", (1, 70), 3, 2.0, 173), 0),
    (_wl("heads_2048_f32", 64, 32, 32, 128, "f32", (24, 36), 3, 1.5, 174), 0),
    (_wl("heads_2048_f32_d64", 64, 32, 32, 64, "f32", (24, 36), 3, 1.5, 175), 0),
    (_wl("heads_2048_window", 64, 32, 32, 128, "bf16", (24, 100), 4, 4.0, 176), 12),
    (_wl("virtual_2048", 64, 32, 8, 128, "f32", (24, 36), 3, 1.5, 177), 0),
    (_wl("virtual_2048_g16", 64, 32, 2, 64, "bf16", (24, 36), 3, 1.5, 178), 0),
    (_wl("crosses_the_walk_s_warp_count", 11, 8, 8, 128, "bf16", (604, 604), 10, 1.0, 179), 0),
]


@pytest.mark.parametrize("launch", ["stream", "layers"])
@pytest.mark.parametrize("wl,window", CASES, ids=lambda x: getattr(x, "name", str(x)))
def test_many_heads_match_the_oracle(cuda_dev, wl, window, launch):
    run = H.Run(wl, cuda_dev, H.random_samples(wl, 80, seed=6), launch=launch, window=window)
    assert run.len_ok, run.len_msgs[:5]
    bad = run.compare()
    assert not bad, bad[:10]


@pytest.mark.parametrize("B,heads", [(57, 32), (73, 25), (300, 40)])
def test_static_scratch_takes_the_same_shape(cuda_dev, B, heads):
    """Bit for bit the regular call's results: the array holds the grid's states."""
    wl = _wl(f"static_{B}", B, heads, heads, 128, "bf16", (30, 40), 2, 1.0, 180)
    pr = S.gen_prompt(wl, 0, cuda_dev)
    outs = []
    for call in (P.dmc_decode_step, P.dmc_decode_step_static_scratch):
        cache = H.cache_for(wl, cuda_dev)
        cache.prefill(0, pr["q0"], pr["k"], pr["v"], pr["cu_seqlens"], pr["max_seqlen"])
        got = []
        for step in range(2):
            x = S.gen_decode(wl, 0, step, cuda_dev)
            out = torch.full_like(x["q"], float("nan"))
            assert call(cache.handle, 0, x["q"].data_ptr(), x["k"].data_ptr(), x["v"].data_ptr(), out.data_ptr(),
                        torch.cuda.current_stream().cuda_stream) == P.DMC_OK
            torch.cuda.synchronize()
            got.append(out)
        assert cache.status()[:2] == (0, 0)
        outs.append(got + [cache.lengths(0)])
    for a, b in zip(*outs):
        assert torch.equal(a, b)
