"""The bounded frontier search (the way an ordinary solve takes) against the CPU oracle where it can go
wrong: every row shape at its edges, quotients too close for one key, a frontier that outgrows its
rows, and the asynchronous entry point.  Exact equality throughout."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from oracle import compute_term as CT
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.helpers import make_instance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    pp.lib()


def same(got, want, what):
    assert got.status == want.status, what
    assert got.beta_ms == want.beta_ms or (np.isinf(got.beta_ms) and np.isinf(want.beta_ms)), what
    assert got.plan() == want.plan(), what


def solve_async(inst):
    import torch
    sol = torch.zeros(22, dtype=torch.float64, device="cuda")
    with pp.Problem.from_instance(inst) as p:
        p.set_stream(torch.cuda.current_stream().cuda_stream)
        for _ in range(2):  # the kernel leaves its counters clean
            p.solve_exact_dev(sol.data_ptr())
        torch.cuda.synchronize()
    rec = pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])
    return pp.Solution(rec.status, rec.beta_ms, rec.m, np.array(rec.cuts), np.array(rec.placement))


@pytest.mark.parametrize("L", [1, 2, 15, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1023])
def test_row_shapes(L):
    # a lane holds 4, 8, 16 or 32 positions, a group 4 to 32 lanes; windows from one layer to the chain
    for i, k in enumerate((2, 4, 6) if L > 300 else (2, 5, 7, 10 if L < 40 else 8)):
        inst = W.random_small(91000 + 10 * L + i, L, k, ties=i == 1, dead_links=0.2 if i == 2 else 0.0)
        cap = inst.node_mem_bytes.copy()
        if L > 8:  # the nodes together hold the chain about twice
            cap = (cap.astype(np.float64) * (2.0 * float(inst.layer_mem_bytes.sum()) / float(cap.sum()))).astype(np.uint64)
        inst = make_instance(inst.layer_out_bits, inst.layer_mem_bytes, cap, inst.bw_kbps, inst.name)
        want = oracle.dp_fact(inst, 8)
        with pp.Problem.from_instance(inst) as p:
            same(p.solve_exact(), want, inst.name)
        same(solve_async(inst), want, inst.name)


def close_instance(seed, L=14, k=6):
    """Quotients that differ only far below a key's resolution: bit counts just below 2^40 that differ by
    single bits, a few bandwidths, and one tiny transfer that stretches the range of the keys."""
    rng = np.random.default_rng(seed)
    bits = (np.uint64((1 << 40) - 200) + rng.integers(0, 150, L).astype(np.uint64))
    bits[int(rng.integers(0, L - 1))] = np.uint64(1)
    mem = rng.integers(2, 6, L).astype(np.uint64)
    cap = rng.integers(9, 16, k).astype(np.uint64)
    bw = W._symmetric(k, lambda n: rng.integers(1, 3, n) * 5_000_000)
    return make_instance(bits, mem, cap, bw, f"close[{seed}]")


def test_quotients_closer_than_a_key():
    for seed in range(12):
        inst = close_instance(seed)
        same(pp.Problem.from_instance(inst).solve_exact(), oracle.dp_fact(inst), inst.name)
        same(solve_async(inst), oracle.dp_fact(inst), inst.name)
        work = np.full(inst.L, 7, np.uint64)
        speed = np.full(inst.k, 3, np.uint32)
        want = CT.dp(inst, work.tolist(), speed.tolist())
        got = pp.solve_exact_compute(inst, work, speed)
        assert got.status == want.status and got.plan() == want.plan(), inst.name
        assert got.beta_ms == want.beta_ms or np.isinf(want.beta_ms)


def test_frontier_that_keeps_every_state():
    # no plan, although the nodes together have room: two layers far apart fit one node only, so no bound
    # ever applies; more rows than the synchronous call's budget, which then takes the dense search
    for L, k in ((12, 8), (9, 16)):
        rng = np.random.default_rng(L)
        mem = np.ones(L, np.uint64)
        mem[1] = mem[L - 2] = 30
        cap = np.full(k, 20, np.uint64)
        cap[k // 2] = 35
        inst = make_instance(rng.integers(1000, 10**6, L).astype(np.uint64), mem, cap,
                             W._symmetric(k, lambda n: rng.integers(1000, 5000, n)), "full")
        want = oracle.dp_fact(inst, 8)
        assert want.status == oracle.INFEASIBLE
        with pp.Problem.from_instance(inst) as p:
            same(p.solve_exact(), want, (L, k))
        same(solve_async(inst), want, (L, k))


def test_threads_and_streams_share_the_device():
    # several solves in flight at once on streams of their own, from several threads
    import threading
    import torch
    insts = [W.config_resnet50_shaped(), W.config_geometric(14, 64, 0), W.config_tiny(), W.config_deeper_cnn()]
    want = [oracle.dp_fact(i, 8) for i in insts]
    bad = []

    def work(inst, w):
        s = torch.cuda.Stream()
        for _ in range(20):
            with pp.Problem.from_instance(inst) as p:
                p.set_stream(s.cuda_stream)
                got = p.solve_exact()
            if got.beta_ms != w.beta_ms or got.plan() != w.plan():
                bad.append(inst.name)

    threads = [threading.Thread(target=work, args=a) for a in zip(insts, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
