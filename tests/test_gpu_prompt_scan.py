"""Prompt compression at the edges of its chunks, row groups and windows (GPU).

A block compresses 128 tokens, split among row groups of 8 to 32 lanes; a
segment may end in its group, in a later one, past the chunk, or many chunks on.
Prompts one below, at and one above the chunk length, segments from one token to
the whole prompt, every row width and type, groups of up to 16 queries (their
importance neurons are read seven at a time after the first) and windows from
one token to the longest, shorter and longer than the segments. Slots, z, counts
and the outputs of a few decode steps against the fp64 oracle, with the
tolerance of the dtype (2e-2 for bf16 caches, 1e-4 for fp32).
"""
import pytest
import torch

from paper_2403_09636_gb300 import DmcCache, synthetic as S
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


def _check(wl, dev, window):
    run = H.Run(wl, dev, H.all_samples(wl), window=window)
    assert run.len_ok, run.len_msgs[:5]
    bad = run.compare()
    assert not bad, bad[:10]


@pytest.mark.parametrize("window", [0, 1, 9, 32])
@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 700])
def test_chunk_edges(cuda_dev, n, dtype, D, window):
    wl = S.Workload(f"scan_{dtype}_{D}_{n}", 1, 2, 3, 3, D, dtype, (n, n), 3, ("choice", (1.0, 4.0, 40.0)),
                    1.0 if dtype == "f32" else 0.5, seed=800 + n + window)
    _check(wl, cuda_dev, window)


@pytest.mark.parametrize("window", [0, 12])
@pytest.mark.parametrize("n", [130, 256, 600])
def test_segments_over_many_chunks(cuda_dev, n, window):
    wl = S.Workload(f"scan_long_{n}", 1, 3, 4, 4, 128, "bf16", (n - 3, n + 3), 3, ("choice", (120.0, 1e6)), 0.5,
                    seed=900 + n)
    _check(wl, cuda_dev, window)


@pytest.mark.parametrize("G", [7, 8, 9, 16])
def test_groups_of_queries(cuda_dev, G):
    wl = S.Workload(f"scan_g{G}", 1, 2, 2 * G, 2, 64, "f32", (150, 200), 2, ("fixed", 5.0), 1.0, seed=950 + G)
    _check(wl, cuda_dev, 0)


@pytest.mark.parametrize("window", [0, 12])
@pytest.mark.parametrize("openings", [(0, 5), (0, 130, 130 + 131 * 128), (0, 128 * 257 + 1)])
def test_openings_hundreds_of_chunks_apart(cuda_dev, openings, window):
    """The next opening is looked for 128 chunks at a time, the last one (window
    grouping) 256: a prompt of 258 chunks, one decoded token that joins the last
    segment. K and V within bf16's 2e-2; z is an fp32 sum over at most ~300 partial
    sums, each rounded to 6e-8 of it: 1e-4 with the omegas' own error."""
    n, D = 128 * 258 - 3, 128
    g = torch.Generator(device=cuda_dev).manual_seed(5)
    k, v = (torch.randn((n + 1, 1, D), generator=g, device=cuda_dev).mul_(0.5).bfloat16() for _ in range(2))
    q = torch.randn((n + 1, 1, D), generator=g, device=cuda_dev).mul_(0.5).bfloat16()
    k[:, :, 0] = k[:, :, 0].abs() + 0.1
    for t in openings:
        k[t, 0, 0] = -1.0
    cache = DmcCache(1, 1, 1, 1, D, torch.bfloat16, 64, 4, n, window=window, device="cuda")
    cu = torch.tensor([0, n], dtype=torch.int32, device=cuda_dev)
    cache.prefill(0, q[:n, :, 0], k[:n], v[:n], cu, n)

    def check(end):
        ends = list(openings[1:]) + [end]
        K, V, z, m = cache.export_heads(0, [0], len(openings) + 1)
        assert int(m[0]) == len(openings)
        for i, (a, b) in enumerate(zip(openings, ends)):
            a = max(a, b - window) if window else a
            w = torch.sigmoid(q[a:b, 0, 0].double())
            kd, vd = k[a:b, 0].double(), v[a:b, 0].double()
            kd[:, 0] = 0
            assert float((K[0, i].double() - (w[:, None] * kd).sum(0) / w.sum()).abs().max()) <= 2e-2
            assert float((V[0, i].double() - (w[:, None] * vd).sum(0) / w.sum()).abs().max()) <= 2e-2
            assert abs(float(z[0, i]) - float(w.sum())) <= 1e-4 * float(w.sum())

    check(n)
    out = torch.empty((1, 1, D), dtype=torch.bfloat16, device=cuda_dev)
    cache.decode(0, q[n:], k[n:], v[n:], out)
    check(n + 1)
    assert cache.status()[:2] == (0, 0)
