"""Window grouping: which prompt rows count (GPU).

A slot is the omega-weighted mean of its segment's last W tokens, so a token more than
W before its segment's end is left out, by its bit in the opening words of its chunk and
the next. Segment ends one below, at and one above W past a token, past its row group,
its 32-token word and its 128-token chunk, prompts that end there, and prompts that
continue a segment; every row that does not count is NaN and must not be seen. Slots
and z against the same means in fp64 (bf16 within 2e-2, fp32 within 1e-4).
"""
import pytest
import torch

from paper_2403_09636_gb300 import DmcCache
from tests import dmc_harness as H

pytestmark = pytest.mark.gpu


def _openings(W):
    ends = sorted({e + d for e in (16, 31, 32, 64, 96, 127, 128, 160, 256, 290) for d in (-W, 0, W - 1, W, W + 1)})
    return [0] + [e for e in ends if e > 0]


@pytest.mark.parametrize("W", [1, 2, 7, 31, 32])
@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
def test_rows_past_the_window_do_not_count(cuda_dev, dtype, D, W):
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device=cuda_dev).manual_seed(W)
    every = _openings(W)
    heads = [every, every[::2], every[::3], [0, 128 + W], [0]]  # the openings of each head
    Hh = len(heads)
    for n, cut in ((128 + W, 0), (290, 0), (300, 0), (300, 40), (300, 128), (413, 271)):
        k, v = (torch.randn((n, Hh, D), generator=g, device=cuda_dev).mul_(0.5) for _ in range(2))
        q0 = torch.randn((n, Hh), generator=g, device=cuda_dev).to(dt)
        k[..., 0] = 1.0
        want = []
        for h, at in enumerate(heads):
            at = [a for a in at if a < n]
            k[at[1:], h, 0] = -1.0
            segs = list(zip(at, at[1:] + [n]))
            for a, b in segs:  # what does not count: in no prompt part's reach (the part ends at `cut` too)
                for t in range(a, b):
                    if b - t > W and not (t < cut < b and cut - t <= W):
                        k[t, h, 1:] = float("nan")
                        v[t, h] = float("nan")
            want.append(segs)
        k, v = k.to(dt), v.to(dt)
        c = DmcCache(1, 1, Hh, Hh, D, dt, 256, 8 * Hh, n, window=W)
        for a, b in ((0, cut), (cut, n)):
            if b > a:
                cu = torch.tensor([0, b - a], dtype=torch.int32, device=cuda_dev)
                c.prefill(0, q0[a:b], k[a:b].contiguous(), v[a:b].contiguous(), cu, b - a)
        assert c.status()[:2] == (0, 0)
        K, V, z, ln = c.export_heads(0, list(range(Hh)), 256)
        w = torch.sigmoid(q0.double())
        kd = k.double()
        kd[..., 0] = 0.0
        for h, segs in enumerate(want):
            assert int(ln[h]) == len(segs)
            for i, (a, b) in enumerate(segs):
                lo = max(a, b - W)
                ws = w[lo:b, h]
                tol = H.TOL[dtype]
                assert abs(float(z[h, i]) - float(ws.sum())) <= tol
                for got, x in ((K, kd), (V, v.double())):
                    ref = (ws[:, None] * x[lo:b, h]).sum(0) / ws.sum()
                    err = float((got[h, i].double() - ref).abs().max())
                    assert err <= tol, (n, cut, h, i, err)
