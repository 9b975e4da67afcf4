"""The search by thresholds at the sizes where it can go wrong: rows of one word and of two, both sides of every line of its
dispatch, many equal terms, terms of nothing, no plan at all, and instances it has to hand over."""
from __future__ import annotations

import contextlib
import time

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from oracle import compute_term as CT
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu


def network(seed, L, k, kind):
    """Nodes that hold a fifth to two thirds of the chain each; every third kind with links of their own each way."""
    inst = W.random_small(seed, L, k, ties=kind == 1, dead_links=0.3 if kind == 2 else 0.0)
    rng = np.random.default_rng(seed)
    total = float(inst.layer_mem_bytes.sum())
    inst.node_mem_bytes[:] = (total * rng.uniform(0.2, 0.67, k)).astype(np.uint64)
    if kind == 3:  # transfers of nothing, and directed links
        inst.layer_out_bits[rng.random(L) < 0.5] = 0
        inst.bw_kbps[:] = rng.integers(1000, 12000, (k, k)) * (1 - np.eye(k, dtype=np.int64))
    if kind == 4:  # hardly room: most have no plan
        inst.node_mem_bytes[:] = (total * rng.uniform(0.2, 2.2, k) / k).astype(np.uint64)
    if kind == 5:  # one value everywhere
        inst.layer_out_bits[:] = 12345
        inst.bw_kbps[:] = 777 * (1 - np.eye(k, dtype=np.int64))
    return inst


def three_nodes(inst):
    """No two nodes hold the chain: where two do, the bounded search is as fast and is the one that runs."""
    total = float(inst.layer_mem_bytes.sum())
    inst.node_mem_bytes[:] = (total * np.random.default_rng(inst.L).uniform(0.2, 0.45, inst.k)).astype(np.uint64)


def rising(seed, L, k):
    """A chain whose memory rises along it, log-normal sizes and links: its optimum takes six nodes and more now and then."""
    rng = np.random.default_rng(seed)
    mem = 64.0 ** (np.arange(L) / L) * (0.8 + 0.4 * rng.random(L))
    bits = np.clip(np.exp(np.log(10.2e6) - 0.28 + 0.75 * rng.standard_normal(L)), 1e5, 1.2e8)
    cap = rng.integers(24 * 10**6, 48 * 10**6, k)
    bw = np.zeros((k, k), np.uint32)
    bw[np.triu_indices(k, 1)] = np.clip(np.exp(np.log(6000) - 0.125 + 0.5 * rng.standard_normal(k * (k - 1) // 2)), 500, 50000)
    return W.Instance(L, k, bits.astype(np.uint64), (mem / mem.sum() * 102_400_000).astype(np.uint64), cap.astype(np.uint64), bw + bw.T, "rising")


def same(got, want):
    assert got.status == want.status and got.plan() == want.plan()
    assert got.beta_ms == want.beta_ms or np.isinf(want.beta_ms)


@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k", [(2, 8), (8, 7), (17, 7), (31, 8), (32, 8), (33, 7), (33, 8), (63, 8), (64, 7), (64, 8), (65, 8), (40, 9)])
def test_transfers_only(L, k, debug):
    build.build()
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        for i in range(18):
            inst = network(120_000 + 100 * L + 10 * k + i, L, k, i % 6)
            want = oracle.dp_fact(inst, 4)
            with pp.Problem.from_instance(inst) as p:
                same(p.solve_exact(), want)
                if i < 6:  # the dense search, which takes every form
                    p.force_generic(1)
                    same(p.solve_exact(), want)


@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k", [(39, 5), (40, 5), (33, 6), (34, 6), (28, 7), (29, 7), (2, 8), (31, 8), (32, 8), (33, 8), (64, 5), (65, 5)])
def test_compute_times(L, k, debug):
    build.build()
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        for i in range(6 if k < 7 else 3):
            inst = network(130_000 + 100 * L + 10 * k + i, L, k, i % 6)
            rng = np.random.default_rng(i)
            work = rng.integers(0, 10**6, L).astype(np.uint64) if i % 3 else np.full(L, 70_000, np.uint64)
            speed = rng.integers(0 if i == 2 else 500, 4000, k).astype(np.uint32)
            same(pp.solve_exact_compute(inst, work, speed), CT.dp(inst, work.tolist(), speed.tolist()))


@pytest.mark.parametrize("L,k", [(24, 9), (33, 10), (64, 10), (50, 11), (20, 12), (50, 12), (64, 12)])
def test_no_work_leaves_the_transfers(L, k):
    """Nothing costs compute: the optimum of Eq. 2."""
    build.build()
    for i in range(8):
        inst = network(140_000 + 100 * L + 10 * k + i, L, k, i % 6)
        if i >= 6:  # many nodes to a plan: with eleven and more the bounded search from the start
            inst.node_mem_bytes[:] = (float(inst.layer_mem_bytes.sum()) * np.random.default_rng(i).uniform(0.12, 0.3, k)).astype(np.uint64)
        want = oracle.dp_fact(inst, 8)
        same(pp.solve_exact_compute(inst, np.zeros(L, np.uint64), np.full(k, 1000, np.uint32)), want)


def test_transfers_only_on_a_stream_of_its_own():
    """A search that takes every SM is for the legacy stream, whose solves run one after another: handles on streams of their own
    go on side by side (four of them took 1.2 times as long as one, by thresholds 3.5 times)."""
    import torch
    build.build()
    insts = [W.config_geometric(8, 48, seed) for seed in range(2, 6)]
    want = [oracle.dp_fact(i, 8) for i in insts]
    streams = [torch.cuda.Stream() for _ in insts]
    sols = [torch.zeros(22, dtype=torch.float64, device="cuda") for _ in insts]
    with contextlib.ExitStack() as stack:
        ps = [stack.enter_context(pp.Problem.from_instance(i)) for i in insts]
        for p, w in zip(ps, want):
            same(p.solve_exact(), w)
            assert pp.debug_thresholds() == 1
        for p, w, s in zip(ps, want, streams):
            p.set_stream(s.cuda_stream)
            same(p.solve_exact(), w)
            assert pp.debug_thresholds() == 0

        def seconds(n):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(100):
                for p, sol in zip(ps[:n], sols):
                    p.solve_exact_dev(sol.data_ptr())
            torch.cuda.synchronize()
            return time.perf_counter() - t0

        times = [(seconds(1), seconds(4)) for _ in range(9)][2:]
        assert np.median([t[1] for t in times]) < 2.5 * np.median([t[0] for t in times]), times
        for sol, w in zip(sols, want):
            got = pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])
            assert got.beta_ms == w.beta_ms and (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == w.plan()
        for p, w in zip(ps, want):
            p.set_stream(0)
            same(p.solve_exact(), w)
            assert pp.debug_thresholds() == 1


# the lines of the dispatch under Eq. 2, on the legacy stream: up to 64 layers and eight nodes, more than a block's round
@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L,k,takes", [(8, 6, 0), (17, 7, 1), (31, 8, 1), (32, 8, 1), (33, 7, 1), (33, 8, 1), (64, 7, 1), (64, 8, 1), (65, 8, 0),
                                       (40, 9, 0)])
def test_which_search_answers(L, k, takes, debug):
    build.build()
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        for kind in (0, 2, 3):
            inst = network(160_000 + 100 * L + 10 * k + kind, L, k, kind)
            three_nodes(inst)
            with pp.Problem.from_instance(inst) as p:
                same(p.solve_exact(), oracle.dp_fact(inst, 4))
            assert pp.debug_thresholds() == takes, kind


# rows of one word and of two
@pytest.mark.parametrize("debug", [False, True])
@pytest.mark.parametrize("L", [24, 50])
def test_what_does_not_fit_is_handed_over(L, debug):
    build.build()
    with library(build.build_debug()) if debug else contextlib.nullcontext():
        # the optimum needs more node sets than a block has room for, or does not
        seen = set()
        for seed in range(12):
            inst = rising(seed, L, 12)
            same(pp.solve_exact_compute(inst, np.zeros(L, np.uint64), np.full(12, 1000, np.uint32)), oracle.dp_fact(inst, 8))
            seen.add(pp.debug_thresholds())
        assert seen == {1, 2}
        # hundreds of quotients within a millionth of each other, in a range that four rounds do not resolve
        for seed in range(4):
            inst = network(seed, L, 8, 0)
            three_nodes(inst)
            rng = np.random.default_rng(seed)
            inst.layer_out_bits[:] = 2**38 + rng.permutation(L)
            inst.layer_out_bits[L // 2] = 2**20
            inst.bw_kbps[:] = (4_000_000 + rng.integers(0, 6, (8, 8))) * (1 - np.eye(8, dtype=np.int64))
            with pp.Problem.from_instance(inst) as p:
                same(p.solve_exact(), oracle.dp_fact(inst, 8))
            assert pp.debug_thresholds() == 2, seed


def no_room(inst):
    inst.node_mem_bytes[:] = np.uint64(float(inst.layer_mem_bytes.sum()) * 0.98 / inst.k)


def one_small_one_slow(inst):
    rng = np.random.default_rng(inst.k)
    inst.layer_out_bits[:] = rng.integers(7_900_000, 8_100_000, inst.L)
    inst.layer_out_bits[inst.L // 2] = 1
    inst.bw_kbps[:] = rng.integers(7800, 8200, (inst.k, inst.k)) * (1 - np.eye(inst.k, dtype=np.int64))
    inst.bw_kbps[1, 3] = inst.bw_kbps[3, 1] = 1


def stack(inst):
    inst.layer_out_bits[: inst.L - 1] = 8_388_608


# takes: whether the search by thresholds is the faster one for such inputs, and therefore asked
@pytest.mark.parametrize("change,L,k,eq1,takes", [(no_room, 50, 7, False, False), (no_room, 50, 8, True, False), (no_room, 50, 5, True, False),
                                                  (one_small_one_slow, 50, 7, False, False), (one_small_one_slow, 50, 5, True, False),
                                                  (one_small_one_slow, 33, 8, True, True), (stack, 33, 7, False, False), (stack, 32, 7, False, True),
                                                  (stack, 50, 5, True, False), (stack, 33, 8, True, True), (stack, 33, 10, True, False),
                                                  (lambda inst: None, 50, 7, False, True), (lambda inst: None, 50, 5, True, True)])
def test_inputs_that_lose_go_to_the_bounded_search(change, L, k, eq1, takes):
    build.build()
    inst = network(150_000 + 100 * L + k, L, k, 0)
    three_nodes(inst)
    change(inst)
    if eq1:
        work, speed = (inst.layer_mem_bytes // np.uint64(1024)).astype(np.uint64), np.random.default_rng(k).integers(500, 1501, k).astype(np.uint32)
        same(pp.solve_exact_compute(inst, work, speed), CT.dp(inst, work.tolist(), speed.tolist()))
    else:
        with pp.Problem.from_instance(inst) as p:
            same(p.solve_exact(), oracle.dp_fact(inst, 4))
    assert pp.debug_thresholds() == (1 if takes else 0)
