"""Calls of several threads whose sizes differ but whose kernel is one: neither takes the other's shared memory away."""
from __future__ import annotations

import threading

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W

pytestmark = pytest.mark.gpu


def in_threads(work, args):
    """work(*a) for every a, at once; what they raised."""
    failed = []

    def run(*a):
        try:
            work(*a)
        except Exception as e:  # noqa: BLE001 - reported by the caller
            failed.append(repr(e))

    threads = [threading.Thread(target=run, args=a) for a in args]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return failed


# (L, k) of one kernel each: rows of 32 positions; rows of 128 and 256
@pytest.mark.parametrize("shapes", [((24, 8), (20, 4)), ((120, 5), (70, 3)), ((250, 4), (140, 2))])
def test_device_batches_of_two_sizes(shapes):
    import torch
    build.build()
    pp.lib()
    B, calls = 8, 2000

    def work(L, k):
        insts = [W.random_small(71000 + 100 * L + i, L, k) for i in range(B)]
        dev = [torch.from_numpy(np.stack([getattr(i, f) for i in insts]).view(t)).cuda() for f, t in (
            ("layer_out_bits", "i8"), ("layer_mem_bytes", "i8"), ("node_mem_bytes", "i8"), ("bw_kbps", "i4"))]
        new = lambda n, t: torch.zeros(n, dtype=t, device="cuda")
        out = [new(B, torch.float64), new(B, torch.int32), new(B * (k - 1), torch.int32), new(B * k, torch.int32), new(B, torch.int8)]
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for _ in range(calls):
            pp.solve_exact_batch_dev(B, L, k, *(t.data_ptr() for t in (*dev, *out)), s.cuda_stream)
        s.synchronize()
        beta, status = out[0].cpu().numpy(), out[4].cpu().numpy()
        for b, inst in enumerate(insts):
            want = oracle.dp_naive(inst)
            assert status[b] == want.status and (beta[b] == want.beta_ms or np.isinf(want.beta_ms)), (L, k, b)

    assert in_threads(work, shapes * 2) == []


@pytest.mark.parametrize("shapes", [((14, 4), (16, 7)), ((100, 10), (70, 11))])  # in one block's shared memory; over several blocks
def test_solves_of_two_sizes(shapes):
    import torch
    build.build()
    pp.lib()

    def work(L, k):
        inst = W.random_small(72000 + L, L, k)
        inst.node_mem_bytes[:] = np.uint64(int(inst.layer_mem_bytes.sum()) // 2 + 1)
        want = oracle.dp_fact(inst, 4)
        sol = torch.zeros(22, dtype=torch.float64, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with pp.Problem.from_instance(inst) as p:
            p.set_stream(s.cuda_stream)
            for _ in range(2000):
                p.solve_exact_dev(sol.data_ptr())
            s.synchronize()
        got = pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])
        assert got.status == want.status and got.beta_ms == want.beta_ms
        assert (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == want.plan()

    assert in_threads(work, shapes * 2) == []
