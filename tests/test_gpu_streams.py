"""Handles on streams that do not wait for the legacy stream: what the library copies to the device is there before
the stream's first launch."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
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
