"""The wait that all warps of a block give up together (GPU).

The warps of the prompt-attention kernel wait through `warp_wait` (dmc_internal.cuh): one
that takes longer than the limit sets DMC_FAULT_WAIT_TIMEOUT and a word that the block
shares, at which every other wait that is not over ends too, so that the kernel drains
and returns. A test-only kernel, built here with the limit at 2 ms, has warps wait on
barriers that nobody arrives at, some of them after one that is complete: all of them
return false within the limit plus scheduling noise (one limit for the block, not one
per wait), the complete ones return true, and the fault bit is set. No tensor-core work
or copy is in flight.
"""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_2403_09636_gb300 import DMC_FAULT_WAIT_TIMEOUT
from paper_2403_09636_gb300 import build as B

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "shared_give_up_probe.cu")
LIMIT_NS = 2_000_000


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("giveup") / "libgiveup.so")
    subprocess.check_call([B.nvcc()] + B.ARCH + B.FLAGS +
                          [f"-DDMC_WAIT_LIMIT_NS={LIMIT_NS}ull", "-shared", SRC, "-o", out])
    lib = C.CDLL(out)
    lib.dmc_shared_give_up_probe.argtypes = [C.c_int, C.c_uint] + [C.c_void_p] * 5
    return lib


@pytest.mark.parametrize("warps,arrived", [(1, 0), (2, 0), (2, 0b01), (12, 0), (12, 0b101101101101), (12, 0xFFF)])
def test_warps_give_up_together(cuda_dev, probe, warps, arrived):
    err = torch.zeros(1, dtype=torch.int32, device=cuda_dev)
    first, second = (torch.full((warps, 32), -1, dtype=torch.int32, device=cuda_dev) for _ in range(2))
    ns = torch.zeros((warps, 32), dtype=torch.int64, device=cuda_dev)
    assert probe.dmc_shared_give_up_probe(warps, arrived, err.data_ptr(), first.data_ptr(), second.data_ptr(),
                                          ns.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    for w in range(warps):
        assert first[w].tolist() == [arrived >> w & 1] * 32
        assert second[w].tolist() == [0] * 32
    assert int(err.item()) == DMC_FAULT_WAIT_TIMEOUT
    # the first wait to give up began within the noise of the others
    assert LIMIT_NS // 2 <= int(ns.min()) and int(ns.max()) < 100 * LIMIT_NS
    assert float(torch.ones(1024, device=cuda_dev).sum()) == 1024.0  # the context is still usable
