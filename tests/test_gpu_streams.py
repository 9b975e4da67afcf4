"""Handles on streams that do not wait for the legacy stream: what the library copies to the device is there before
the stream's first launch."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from oracle import random_plans as OR
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    pp.lib()


def record(sol):
    return pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])


@pytest.mark.parametrize("mode", [-1, 0])  # the bounded search; the dense one, whose tables are copied by its first run
def test_first_calls_of_new_handles(mode):
    import torch
    s = torch.cuda.Stream()
    sol = torch.zeros(22, dtype=torch.float64, device="cuda")
    for i in range(12):
        inst = W.random_small(95000 + i, 40 + 7 * i, 7 + i % 3)
        inst.node_mem_bytes[:] = np.uint64(int(inst.layer_mem_bytes.sum()) // 3 + 1)
        nseg, ends, nodes = W.random_plans(inst, 200, seed=i, invalid_fraction=0.2)
        want, scored = oracle.dp_fact(inst, 4), oracle.eval_plans(inst, nseg, ends, nodes)
        dev = [torch.from_numpy(a).cuda() for a in (nseg, ends, nodes)]
        beta = torch.zeros(200, dtype=torch.float64, device="cuda")
        stat = torch.zeros(200, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        with pp.Problem.from_instance(inst) as p:
            p.force_generic(mode)
            p.set_stream(s.cuda_stream)
            if i % 2:
                p.solve_exact_dev(sol.data_ptr())
            p.eval_plans_dev(200, *(a.data_ptr() for a in dev), beta.data_ptr(), stat.data_ptr())
            if not i % 2:
                p.solve_exact_dev(sol.data_ptr())
            s.synchronize()
        got = record(sol)
        assert got.status == want.status and (np.isinf(want.beta_ms) or got.beta_ms == want.beta_ms)
        assert (got.m, tuple(got.cuts[: max(got.m - 1, 0)]), tuple(got.placement[: got.m])) == want.plan()
        assert np.array_equal(beta.cpu().numpy(), scored[0]) and np.array_equal(stat.cpu().numpy(), scored[1])


def test_first_calls_over_plans_are_plain_launches():
    # nothing is allocated, so that a first call can be recorded into a graph, and the tables are there for it
    import torch
    inst = W.random_small(96000, 61, 9)
    inst.node_mem_bytes[:] = np.uint64(int(inst.layer_mem_bytes.sum()) // 3 + 1)
    B = 700
    nseg, ends, nodes = W.random_plans(inst, B, seed=4, invalid_fraction=0.2)
    off, e16, n8 = W.pack_plans(nseg, ends, nodes)
    want = oracle.eval_plans(inst, nseg, ends, nodes)
    draws = np.random.default_rng(3).integers(0, 2**32, size=(B, 2 * inst.k), dtype=np.uint64).astype(np.uint32)
    drawn = OR.random_plans(inst, draws)
    dev = [torch.from_numpy(a.view("i%d" % a.itemsize) if a.itemsize > 1 else a).cuda()
           for a in (nseg, ends, nodes, off, e16, n8, draws)]
    beta = torch.zeros(B, dtype=torch.float64, device="cuda")
    stat = torch.zeros(B, dtype=torch.uint8, device="cuda")
    out = (torch.zeros(B, dtype=torch.uint8, device="cuda"), torch.zeros((B, inst.k), dtype=torch.int32, device="cuda"),
           torch.zeros((B, inst.k), dtype=torch.int32, device="cuda"))
    ptr = lambda *t: [x.data_ptr() for x in t]
    calls = {"eval": lambda p: p.eval_plans_dev(B, *ptr(*dev[:3], beta, stat)),
             "packed": lambda p: p.eval_plans_packed_dev(B, e16.size, *ptr(dev[0], *dev[3:6], beta, stat)),
             "random": lambda p: p.random_plans_dev(B, *ptr(dev[6], *out))}
    s = torch.cuda.Stream()

    def check(name):
        torch.cuda.synchronize()
        if name == "random":
            assert [t.cpu().numpy().tolist() for t in out] == list(drawn)
        else:
            assert np.array_equal(beta.cpu().numpy(), want[0]) and np.array_equal(stat.cpu().numpy(), want[1])
        for t in (beta, stat, *out):
            t.zero_()
        torch.cuda.synchronize()

    for name, call in calls.items():
        for stream in (0, s.cuda_stream):
            with pp.Problem.from_instance(inst) as p:
                p.set_stream(stream)
                pp.debug_fail_alloc(1)  # the next allocation would fail
                try:
                    call(p)
                finally:
                    pp.debug_fail_alloc(0)
                check(name)
        with pp.Problem.from_instance(inst) as p:
            p.set_stream(s.cuda_stream)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                call(p)
                call(p)
            for _ in range(2):
                g.replay()
                check(name)
            del g
            call(p)  # the handle does not live on the graph's memory
            check(name)


@pytest.mark.parametrize("L,k,mode,workspace", [(12, 6, -1, False), (50, 10, -1, False), (90, 12, -1, False), (337, 9, -1, False),
                                                (50, 10, 0, False), (60, 9, 0, True), (100, 14, -1, True)])
def test_handle_that_meets_its_stream_in_a_recording(L, k, mode, workspace):
    # created before, used for the first time while a graph is recorded: nothing of the handle belongs to the graph
    import torch
    inst = W.random_small(97000 + L, L, k)
    inst.node_mem_bytes[:] = np.uint64(int(inst.layer_mem_bytes.sum()) // 3 + 1)
    want = oracle.dp_fact(inst, 8)
    nseg, ends, nodes = W.random_plans(inst, 300, seed=L, invalid_fraction=0.2)
    scored = oracle.eval_plans(inst, nseg, ends, nodes)
    dev = [torch.from_numpy(a).cuda() for a in (nseg, ends, nodes)]
    sol = torch.zeros(22, dtype=torch.float64, device="cuda")
    beta = torch.zeros(300, dtype=torch.float64, device="cuda")
    stat = torch.zeros(300, dtype=torch.uint8, device="cuda")

    def check():
        torch.cuda.synchronize()
        got = record(sol)
        assert got.status == want.status and got.beta_ms == want.beta_ms
        assert (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == want.plan()
        assert np.array_equal(beta.cpu().numpy(), scored[0]) and np.array_equal(stat.cpu().numpy(), scored[1])
        for t in (sol, beta, stat):
            t.zero_()
        torch.cuda.synchronize()

    def calls(p):
        p.solve_exact_dev(sol.data_ptr())
        p.eval_plans_dev(300, *(a.data_ptr() for a in dev), beta.data_ptr(), stat.data_ptr())

    other = torch.cuda.Stream()
    for first_on in (None, 0, other.cuda_stream):
        with pp.Problem.from_instance(inst) as p:
            p.force_generic(mode)
            if workspace:
                p.set_workspace(torch.empty(p.workspace_bytes(), dtype=torch.uint8, device="cuda"))
            if first_on is not None:  # and the recording begins while these calls may still be running
                p.set_stream(first_on)
                calls(p)
                if first_on == 0:
                    torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                p.set_stream(torch.cuda.current_stream().cuda_stream)
                calls(p)
            for _ in range(3):
                g.replay()
                check()
            del g
            s = torch.cuda.Stream()
            p.set_stream(s.cuda_stream)
            calls(p)
            check()
            got = p.solve_exact()
            assert got.beta_ms == want.beta_ms and got.plan() == want.plan()
