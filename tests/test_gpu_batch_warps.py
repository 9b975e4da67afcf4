"""The batched search an instance to a warp, at sizes that the library's own rule sends there (the smallest of every shape, and
more instances than warps): against the oracle, on close, extreme and equal quotients and on instances beyond the limits."""
from __future__ import annotations

import contextlib

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from tests.test_gpu_batch_dispatch import FIELDS, device_batch, pool
from tests.test_gpu_batch_lanes import check
from tests.test_gpu_batch_ranking import extreme_instances
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu


# rows of windows of every length (those beyond 15 layers lie in shared memory), node sets that fill trips and that do not
@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k,B", [(1, 8, 900), (2, 8, 900), (5, 7, 900), (12, 7, 900), (13, 7, 2000), (14, 8, 900), (15, 8, 1300), (16, 8, 1300),
                                   (17, 8, 1700), (24, 8, 4096), (25, 8, 1100), (25, 7, 1600), (31, 8, 7200), (32, 8, 1100), (32, 7, 1600),
                                   (3, 6, 1800), (8, 6, 1800), (11, 6, 1800), (24, 6, 4097), (25, 6, 3000)])
def test_an_instance_to_a_warp(L, k, B, debug):
    build.build()
    insts = pool(L, k) + (extreme_instances(L, k) if L > 1 else [])
    want = [oracle.dp_naive(i) for i in insts]
    pick = np.random.default_rng(B).permutation(B) % len(insts)
    bits, mem, cap, bw = (np.stack([getattr(i, f) for i in insts])[pick] for f in FIELDS)
    beyond = np.arange(B) % 89 == 17
    bits[beyond, L - 1] = np.uint64(1) << np.uint64(40)   # the smallest transfer refused
    wraps = np.arange(B) % 89 == 20
    mem[wraps] = np.uint64(1) << np.uint64(63)            # the 64-bit sum of the memory wraps
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        assert pp.debug_batch_route(B, L, k) == 0
        got = device_batch(L, k, [bits, mem, cap, bw])
    for b in range(B):
        if beyond[b] or (wraps[b] and L > 1):
            assert got.status[b] == pp.PP_ERR_LIMIT and got.m[b] == 0 and np.isinf(got.beta_ms[b]), b
            assert (got.cuts[b] == -1).all() and (got.placement[b] == -1).all(), b
        elif not wraps[b]:
            check(got, b, want[pick[b]])
