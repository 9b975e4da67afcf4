"""The batched search an instance to a warp, at sizes that the library's own rule sends there (the smallest of every shape, and
more instances than warps): against the oracle, on close, extreme and equal quotients and on instances beyond the limits."""
from __future__ import annotations

import contextlib

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.test_gpu_batch_dispatch import FIELDS, device_batch, pool
from tests.test_gpu_batch_lanes import check
from tests.test_gpu_batch_ranking import extreme_instances
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu


# rows of windows of every length (those beyond 15 layers lie in shared memory), node sets that fill trips and that do not
@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k,B", [(1, 8, 900), (2, 8, 900), (5, 7, 900), (9, 8, 900), (12, 7, 1700), (13, 7, 2100), (14, 8, 1500), (15, 8, 1800), (16, 8, 1800),
                                   (17, 8, 2000), (24, 8, 4096), (25, 8, 1500), (25, 7, 2000), (31, 8, 7200), (32, 8, 1500), (32, 7, 2000),
                                   (3, 6, 1800), (8, 6, 4097), (11, 6, 4097), (24, 6, 4097), (25, 6, 4097)])
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
        assert pp.debug_batch_route(B, L, k) == 32
        got = device_batch(L, k, [bits, mem, cap, bw])
    for b in range(B):
        if beyond[b] or (wraps[b] and L > 1):
            assert got.status[b] == pp.PP_ERR_LIMIT and got.m[b] == 0 and np.isinf(got.beta_ms[b]), b
            assert (got.cuts[b] == -1).all() and (got.placement[b] == -1).all(), b
        elif not wraps[b]:
            check(got, b, want[pick[b]])


def close_quotients(L, k, B, seed=4):
    """Chains and links that are nearly alike, beside one transfer of a bit and one link of 1 kbit/s: hundreds of quotients lie
    within a hundredth of the range of all, on its logarithm a thousandth."""
    rng = np.random.default_rng(seed)
    upper = np.triu_indices(k, 1)
    links = np.rint(4e6 * (1 + 0.01 * rng.random((B, len(upper[0])))))
    links[np.arange(B), rng.integers(0, links.shape[1], B)] = 1
    bw = np.zeros((B, k, k), np.uint32)
    bw[:, upper[0], upper[1]] = links
    bits = (2.0**38 * (1 + 0.005 * rng.random((B, L)))).astype(np.uint64)
    bits[:, L // 2] = 1
    mem = rng.integers(10**6, 4 * 10**7, (B, L)).astype(np.uint64)
    cap = (rng.integers(4 * 10**7, 16 * 10**7, (B, k)) * max(1.0, L / (3.0 * k))).astype(np.uint64)
    return [bits, mem, cap, bw + bw.transpose(0, 2, 1)]


@pytest.mark.parametrize("L,k,B", [(24, 8, 2100), (32, 7, 2100)])
def test_close_quotients_are_not_walked_one_by_one(L, k, B):
    """The time of a batch of close quotients beside one of spread ones: three to five times as much where every quotient between the bound
    and the optimum is a step of its own, a third more by bisection."""
    import torch
    build.build()
    close = close_quotients(L, k, B)
    spread = [a.copy() for a in close]
    rng = np.random.default_rng(5)
    spread[0][:] = rng.integers(10**5, 2 * 10**7, (B, L))
    upper = np.triu_indices(k, 1)
    spread[3][:] = 0
    spread[3][:, upper[0], upper[1]] = rng.integers(1000, 12001, (B, len(upper[0])))
    spread[3] += spread[3].transpose(0, 2, 1)
    assert pp.debug_batch_route(B, L, k) == 32
    for arrays in (close, spread):
        got = device_batch(L, k, arrays)
        for b in range(0, B, 61):
            check(got, b, oracle.dp_naive(W.Instance(L, k, *(a[b] for a in arrays), "close")))
    stream = torch.cuda.current_stream().cuda_stream

    def call(arrays):
        dev = [torch.from_numpy(a.view(f"i{a.dtype.itemsize}")).cuda() for a in map(np.ascontiguousarray, arrays)]
        new = lambda n, t: torch.empty(n, dtype=t, device="cuda")
        out = [new(B, torch.float64), new(B, torch.int32), new(B * (k - 1), torch.int32), new(B * k, torch.int32), new(B, torch.int8)]
        return lambda: pp.solve_exact_batch_dev(B, L, k, *(t.data_ptr() for t in (*dev, *out)), stream)

    calls, times = [call(close), call(spread)], [[], []]
    for turn in range(12):
        for f, t in zip(calls, times):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            f()
            ev[0].record()
            for _ in range(4):
                f()
            ev[1].record()
            ev[1].synchronize()
            if turn >= 2:
                t.append(ev[0].elapsed_time(ev[1]))
    assert np.median(times[0]) < 2.5 * np.median(times[1]), [np.median(t) for t in times]
