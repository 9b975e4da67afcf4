"""Instances whose quotients lie closer together than a key resolves and whose frontier no bound thins out: a
synchronous solve leaves the second search, which would be one block's, to the dense one."""
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


def close_instance(L, k, seed):
    rng = np.random.default_rng(seed)
    bits = np.uint64((1 << 40) - 4000) + rng.integers(0, 3000, L).astype(np.uint64)
    bits[int(rng.integers(0, L - 1))] = np.uint64(1)  # stretches the range of the keys
    bw = np.full((k, k), 5_000_000, np.uint32)
    np.fill_diagonal(bw, 0)
    # every node is needed, so that the first complete plans come on the last level
    return make_instance(bits, np.full(L, 10), np.full(k, 10 * L // k + 10), bw, f"close[{L},{k}]")


# frontiers below and above the line from which the dense search takes over; rows of 2, 4, 8 and 16 positions a lane
@pytest.mark.parametrize("L,k", [(20, 9), (30, 11), (60, 12), (100, 13), (140, 12), (260, 11)])
def test_second_search_of_a_wide_frontier(L, k):
    import torch
    for seed in range(2):
        inst = close_instance(L, k, seed)
        want = oracle.dp_fact(inst, 8)
        assert want.status == oracle.OK
        sol = torch.zeros(22, dtype=torch.float64, device="cuda")
        with pp.Problem.from_instance(inst) as p:
            s = torch.cuda.Stream()
            p.set_stream(s.cuda_stream)
            for _ in range(2):
                got = p.solve_exact()
                assert got.beta_ms == want.beta_ms and got.plan() == want.plan()
            # by block 0 alone 2.5 ms at L = 60, k = 12 and 12 at L = 100, k = 13; both searches together below 0.5
            assert p.last_solve_profile().ms_total < 2.0
            p.solve_exact_dev(sol.data_ptr())
            torch.cuda.synchronize()
        got = pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])
        assert got.status == pp.PP_OK and got.beta_ms == want.beta_ms
        assert (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == want.plan()


def test_second_search_under_eq1():
    inst = close_instance(30, 12, 3)
    work, speed = np.full(inst.L, 7, np.uint64), np.full(inst.k, 3, np.uint32)
    want = CT.dp(inst, work.tolist(), speed.tolist())
    got = pp.solve_exact_compute(inst, work, speed)
    assert got.status == want.status and got.plan() == want.plan() and got.beta_ms == want.beta_ms
