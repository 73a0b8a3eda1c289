"""Which decode launches may overlap the launch before them (CPU).

A decode launch with the programmatic attribute starts while the kernel before it on
its stream still runs, and reads its layers' slot counts, page table and pages before
it waits for it. The rule (csrc/dmc_overlap.h, compiled here for the host) is run over
sequences of calls and compared with what is safe: the call before, in the order of
the calls, was a decode on the same stream of other layers than this one's.
"""
import ctypes as C
import itertools
import os
import random
import subprocess

import pytest

from paper_2403_09636_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "overlap_rule.cpp")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("overlap") / "liboverlap.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-shared", "-fPIC", "-I", B.CSRC, SRC, "-o", out])
    lib = C.CDLL(out)

    def run(calls):  # (first layer, layers, stream, the handle stands for one stream)
        n = len(calls)
        cols = [(t * n)(*[c[i] for c in calls]) for i, t in enumerate((C.c_int, C.c_int, C.c_longlong, C.c_int))]
        may = (C.c_int * n)()
        lib.dmc_overlap_rule(n, *cols, may)
        return [bool(x) for x in may]

    return run


def _safe(before, call):
    if before is None or before[1] == 0 or call[1] == 0:
        return False
    other = not set(range(before[0], before[0] + before[1])) & set(range(call[0], call[0] + call[1]))
    return bool(other and before[2] == call[2] and call[3])


def _check(rule, calls):
    want = [_safe(b, c) for b, c in zip([None] + calls, calls)]
    assert rule(calls) == want, calls


def test_a_prompt_on_another_stream_in_between(rule):
    """prefill(1, B), decode(0, A), decode(1, B): the last one's predecessor on B is
    the prompt of its own layer."""
    A, Bs = 16, 32
    assert rule([(0, 0, Bs, 1), (0, 1, A, 1), (1, 1, Bs, 1)]) == [False, False, False]
    assert rule([(0, 0, A, 1), (0, 1, A, 1), (1, 1, A, 1)]) == [False, False, True]


def test_single_layers_on_two_streams(rule):
    calls = [(layer, n, s, 1) for layer, n in ((0, 0), (0, 1), (1, 1)) for s in (16, 32)]
    for seq in itertools.product(calls, repeat=4):
        _check(rule, list(seq))


def test_a_handle_for_many_streams_never_overlaps(rule):
    assert rule([(0, 1, 2, 0), (1, 1, 2, 0), (0, 1, 2, 0)]) == [False] * 3


def test_random_sequences_of_single_layers(rule):
    rng = random.Random(3)
    for _ in range(300):
        _check(rule, [(rng.randrange(4), rng.choice((0, 1, 1, 1)), rng.choice((0, 16)), rng.random() < 0.9)
                      for _ in range(20)])


def test_ranges_of_layers_have_to_be_apart(rule):
    """decode(1), then one launch over layers 0 and 1: it may not read layer 1's counts
    while the first publishes them."""
    assert rule([(1, 1, 16, 1), (0, 2, 16, 1), (2, 2, 16, 1), (0, 2, 16, 1)]) == [False, False, True, True]


def test_random_sequences_of_ranges(rule):
    rng = random.Random(4)
    for _ in range(500):
        _check(rule, [(lambda lo: (lo, rng.choice((0, 1, 1, 2, 3)), rng.choice((0, 16)), rng.random() < 0.9))
                      (rng.randrange(5)) for _ in range(20)])
