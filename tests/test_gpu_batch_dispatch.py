"""The batched search on both sides of every line of its dispatch: batches of one and two waves of blocks, and the
batches beyond them that go an instance to a lane or to a warp, over the row widths of all paths."""
from __future__ import annotations

import contextlib

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from paper_2210_12219_b200.binding import BatchSolution
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu

FIELDS = ("layer_out_bits", "layer_mem_bytes", "node_mem_bytes", "bw_kbps")


def pool(L, k, n=37):
    """Networks of every kind the search knows, one direction of the links unlike the other in some."""
    rng = np.random.default_rng(1000 * L + k)
    insts = []
    for i in range(n):
        a = W.random_small(93000 + 100 * L + i, L, k, tight=(i % 3 == 1), ties=(i % 3 == 2), dead_links=0.25 if i % 4 == 3 else 0.0)
        bw = a.bw_kbps
        if i % 5 == 4:
            bw = rng.integers(1000, 12000, size=(k, k)).astype(np.uint32)
            np.fill_diagonal(bw, 0)
        insts.append(W.Instance(L, k, a.layer_out_bits, a.layer_mem_bytes, a.node_mem_bytes, bw, f"dispatch[{i}]"))
    return insts


def device_batch(L, k, arrays):
    """The batch through the device-pointer entry point, its results laid out as the host variant's."""
    import torch
    B = arrays[0].shape[0]
    dev = [torch.from_numpy(a.view(f"i{a.dtype.itemsize}")).cuda() for a in map(np.ascontiguousarray, arrays)]
    new = lambda n, t: torch.empty(n, dtype=t, device="cuda")
    beta, m, cuts = new(B, torch.float64), new(B, torch.int32), new((B, max(k - 1, 1)), torch.int32)
    place, status = new((B, k), torch.int32), new(B, torch.int8)
    pp.solve_exact_batch_dev(B, L, k, *(t.data_ptr() for t in (*dev, beta, m, cuts, place, status)),
                             torch.cuda.current_stream().cuda_stream)
    return BatchSolution(*(t.cpu().numpy() for t in (beta, m, cuts[:, : k - 1], place, status)))


# device batches of at most three (two for k = 8 from 29 layers on) blocks an SM of 148, of up to twice as many, for k <= 6
# in narrow blocks, of up to twice as many again, and larger ones; longer chains, which always go an instance to a block
@pytest.mark.parametrize("L,k,debug", [(1, 4, False), (7, 8, False), (16, 3, False), (16, 8, False), (17, 6, False), (24, 7, False),
                                       (25, 7, False), (24, 8, True), (32, 4, True), (32, 8, False), (45, 5, True),
                                       (66, 4, False), (130, 3, False), (258, 2, False)])
def test_every_path_gives_the_oracles_plans(L, k, debug):
    build.build()
    insts = pool(L, k)
    want = [oracle.dp_naive(i) for i in insts]
    beyond = 11  # this one has a transfer beyond the limits
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        # the last one is more than the host variant works on in place: it goes an instance to a lane or to a warp
        for B in (63, 64, 296, 297, 444, 445, 888, 889, 1332, 1333, max(1800, (1 << 20) // (16 * L + 4 * k * (k + 3)) + 45)):
            pick = np.arange(B) % len(insts)
            arrays = [np.stack([getattr(i, f) for i in insts])[pick].copy() for f in FIELDS]
            flagged = pick == beyond
            arrays[0][flagged, L - 1] = np.uint64(1) << np.uint64(41)
            got = device_batch(L, k, arrays) if B < 1800 else pp.solve_exact_batch(L, k, *arrays)
            if B in (64, 889):
                host = pp.solve_exact_batch(L, k, *arrays)
                for x, y in zip((got.beta_ms, got.m, got.cuts, got.placement, got.status),
                                (host.beta_ms, host.m, host.cuts, host.placement, host.status)):
                    assert np.array_equal(x, y)
            for b in list(range(min(B, 80))) + list(range(80, B, 29)) + [B - 1]:
                if flagged[b]:
                    assert got.status[b] == pp.PP_ERR_LIMIT and got.m[b] == 0 and np.isinf(got.beta_ms[b]), (B, b)
                    continue
                w = want[pick[b]]
                assert got.status[b] == w.status and got.plan(b) == w.plan(), (B, b)
                assert got.beta_ms[b] == w.beta_ms or np.isinf(w.beta_ms), (B, b)
            for x in (got.beta_ms, got.m, got.status):  # and all the others like the first of their kind
                assert np.array_equal(x, x[pick])


# narrow blocks on rows that take them two rounds to stage, and batches of more instances than blocks, which take several
# in turn (narrow and wide ones)
@pytest.mark.parametrize("L,k,B,threads", [(200, 3, 445, 192), (256, 2, 445, 192), (193, 3, 900, 192), (45, 6, 2401, 192), (45, 4, 4801, 192),
                                           (45, 7, 2401, 384)])
@pytest.mark.parametrize("debug", [False, True])
def test_long_rows_and_blocks_of_several_instances(L, k, B, threads, debug):
    import torch
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    insts = pool(L, k)
    want = [oracle.dp_naive(i) for i in insts]
    pick = np.random.default_rng(B).permutation(B) % len(insts)
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        assert pp.debug_batch_route(B, L, k, sms=sms) == threads
        got = device_batch(L, k, [np.stack([getattr(i, f) for i in insts])[pick] for f in FIELDS])
    for b in range(B):
        w = want[pick[b]]
        assert got.status[b] == w.status and got.plan(b) == w.plan(), b
        assert got.beta_ms[b] == w.beta_ms or np.isinf(w.beta_ms), b
