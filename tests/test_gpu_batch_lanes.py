"""The batched search an instance to a lane, at sizes that the library's own rule sends there: its quotients and the ranking
of extreme and close ones, instances beyond the limits, and batches that are worked off in pieces which share the scratch tables."""
from __future__ import annotations

import contextlib

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.test_gpu_batch_dispatch import FIELDS, device_batch
from tests.test_gpu_batch_ranking import extreme_instances
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu


def lanes(B, L, k):
    import torch
    return pp.debug_batch_route(B, L, k, sms=torch.cuda.get_device_properties(0).multi_processor_count) == 0  # 32: to a warp


def smallest_for_lanes(L, k):
    """The smallest batch from which on this shape goes an instance to a lane, made to end inside a group of 32."""
    B = next(B for B in range(64, 1 << 16) if lanes(B, L, k))
    B += 32 - B % 32 + 13
    assert lanes(B, L, k)
    return B


def check(got, b, want):
    assert got.status[b] == want.status and got.plan(b) == want.plan(), b
    assert got.beta_ms[b] == want.beta_ms or np.isinf(want.beta_ms), b
    assert (got.cuts[b, max(want.m - 1, 0):] == -1).all() and (got.placement[b, want.m:] == -1).all(), b


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def near_middles(n, rng):
    """Pairs whose quotient lies as near to the middle of two doubles as one with this bandwidth can, on either side."""
    bits, kbps = [], []
    for b in rng.integers(1 << 12, 1 << 23, n) * 2 + 1:
        b = int(b)
        for sign in (1, -1):
            x = int(rng.integers(1 << 38, 1 << 39))
            shift = 52 - ((x // b).bit_length() - 1)  # the quotient times 2^shift has 53 bits before the point
            x += (sign * pow(2, -(shift + 1), b) - x) % b  # 2^(shift + 1) x = sign modulo b: a middle and 1 / (2 b) of a unit
            bits.append(x)
            kbps.append(b)
    return bits, kbps


def test_quotients_are_correctly_rounded():
    rng = np.random.default_rng(5)
    edges = [0, 1, 2, 3, (1 << 24) - 1, 1 << 24, (1 << 24) + 1, (1 << 39) - 1, 1 << 39, (1 << 40) - 2, (1 << 40) - 1]
    links = [1, 2, 3, 5, 7, (1 << 12) - 1, 1 << 12, (1 << 23) - 1, 1 << 23, (1 << 23) + 1, (1 << 24) - 2, (1 << 24) - 1]
    edge = np.array([(x, b) for x in edges for b in links], dtype=np.uint64)
    small = np.array([(x, b) for x in range(600) for b in range(1, 600)], dtype=np.uint64)
    hard = np.array(near_middles(100_000, rng), dtype=np.uint64).T
    n = 1 << 23
    whole = np.stack([rng.integers(0, 1 << 40, n, dtype=np.uint64), rng.integers(1, 1 << 24, n, dtype=np.uint64)], axis=1)
    spread = np.stack([np.exp2(rng.uniform(0, 40, n)).astype(np.uint64), np.exp2(rng.uniform(0, 24, n)).astype(np.uint64)], axis=1)
    spread[:, 0] = np.minimum(spread[:, 0], (1 << 40) - 1)
    spread[:, 1] = np.minimum(spread[:, 1], (1 << 24) - 1)
    for pairs in (edge, small, hard, whole, spread):
        by_reciprocal, divided = pp.debug_quotients(pairs[:, 0], pairs[:, 1])
        want = pairs[:, 0].astype(np.float64) / pairs[:, 1].astype(np.float64)
        assert np.array_equal(by_reciprocal.view(np.uint64), divided.view(np.uint64))
        assert np.array_equal(by_reciprocal.view(np.uint64), want.view(np.uint64))
    for x, b in ((1 << 40, 1), (1, 0), (1, 1 << 24)):
        with pytest.raises(pp.PPError) as e:
            pp.debug_quotients([x], [b])
        assert e.value.status == pp.PP_ERR_LIMIT


@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k", [(7, 3), (8, 7), (9, 2), (17, 5), (24, 8), (31, 6), (32, 8)])
def test_extreme_and_close_quotients(L, k, debug):
    insts = extreme_instances(L, k)
    want = [oracle.dp_naive(i) for i in insts]
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        B = smallest_for_lanes(L, k)
        pick = np.random.default_rng(B).permutation(B) % len(insts)
        got = device_batch(L, k, [np.stack([getattr(i, f) for i in insts])[pick] for f in FIELDS])
    for b in range(B):
        check(got, b, want[pick[b]])


@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k", [(12, 4), (7, 6), (32, 8)])
def test_instances_beyond_the_limits(L, k, debug):
    insts = [W.random_small(62000 + 100 * L + i, L, k) for i in range(80)]
    want = [oracle.dp_naive(i) for i in insts]
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        B = smallest_for_lanes(L, k)
        pick = np.arange(B) % len(insts)
        bits, mem, cap, bw = (np.stack([getattr(i, f) for i in insts])[pick] for f in FIELDS)
        bits[17::80, L - 2] = np.uint64(1) << np.uint64(40)   # the smallest transfer refused
        mem[20::80, :2] = np.uint64(1) << np.uint64(63)       # the 64-bit sum of the memory wraps
        bw[23::80, 1, k - 1] = np.uint32(1) << np.uint32(24)  # the smallest bandwidth refused
        bw[24::80, 1, 1] = np.uint32(1) << np.uint32(24)      # likewise where no link is
        got = device_batch(L, k, [bits, mem, cap, bw])
    for b in range(B):
        if b % 80 in (17, 20, 23, 24):
            assert got.status[b] == pp.PP_ERR_LIMIT and got.m[b] == 0 and np.isinf(got.beta_ms[b]), b
            assert (got.cuts[b] == -1).all() and (got.placement[b] == -1).all(), b
        else:
            check(got, b, want[pick[b]])


# 4096 instances share the scratch tables at a time: whole pieces, and a last one of a few instances or of one, over all widths
# of a row (with six nodes and more the lanes take one piece at most)
@pytest.mark.parametrize("L,k,B,debug", [(9, 4, 4096 + 45, False), (8, 5, 2 * 4096 + 1, True), (24, 5, 4097, False), (32, 5, 4097, True),
                                         (24, 6, 4096, False), (5, 5, 4096, False)])
def test_pieces_one_after_another(L, k, B, debug):
    insts = [W.random_small(66000 + i, L, k, tight=(i % 3 == 1), ties=(i % 7 == 2), dead_links=0.25 if i % 4 == 3 else 0.0)
             for i in range(B)]
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        assert lanes(B, L, k)
        got = device_batch(L, k, [np.stack([getattr(i, f) for i in insts]) for f in FIELDS])
    for b in range(B):
        check(got, b, oracle.dp_naive(insts[b]))
