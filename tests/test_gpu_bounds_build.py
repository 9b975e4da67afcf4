"""The bounds-checking build: every kernel with tables of its own does check its accesses there, runs clean, and the
normal build checks nothing."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from oracle import compute_term as CT
from oracle import random_plans as OR
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu

PRUNE, BATCH, MATCH, EVAL, RANDOM = range(5)


def run_everything():
    """One call of every kind, checked against the oracles -> checks made by the kernels of each source."""
    for kernel in range(5):
        pp.debug_bounds_checks(kernel)
    seen = {}
    # the bounded search: in shared memory, one cluster, the whole grid; rows of 2, 4, 8 and 16 positions a lane
    for inst in (W.config_tiny(), W.config_resnet50_shaped(), W.random_small(98001, 70, 9), W.random_small(98002, 150, 8),
                 W.random_small(98003, 300, 9)):
        cap = inst.node_mem_bytes.astype(np.float64)
        inst.node_mem_bytes[:] = (cap * max(1.0, 2.0 * float(inst.layer_mem_bytes.sum()) / cap.sum())).astype(np.uint64)
        want = oracle.dp_fact(inst, 4)
        with pp.Problem.from_instance(inst) as p:
            got = p.solve_exact()  # a recorded violation would raise PP_ERR_CUDA
        assert got.status == want.status and got.plan() == want.plan(), inst.name
        n = pp.debug_bounds_checks(PRUNE)
        seen[inst.name, inst.L] = n
    inst = W.config_geometric(9, 64, 4)
    work = (inst.layer_mem_bytes // np.uint64(1024)).astype(np.uint64)
    speed = (1000 + 37 * np.arange(inst.k)).astype(np.uint32)
    want = CT.dp(inst, work.tolist(), speed.tolist())
    got = pp.solve_exact_compute(inst, work, speed)
    assert got.status == want.status and got.plan() == want.plan()
    seen["eq1"] = pp.debug_bounds_checks(PRUNE)
    insts = [W.random_small(98100 + i, 45, 5) for i in range(8)]
    got = pp.solve_exact_batch(45, 5, *(np.stack([getattr(i, a) for i in insts]) for a in (
        "layer_out_bits", "layer_mem_bytes", "node_mem_bytes", "bw_kbps")))
    for b, i in enumerate(insts):
        want = oracle.dp_naive(i)
        assert got.status[b] == want.status and got.plan(b) == want.plan()
    seen["batch"] = pp.debug_bounds_checks(BATCH)
    draws = np.random.default_rng(5).integers(0, 2**32, size=(12, inst.k), dtype=np.uint64).astype(np.uint32)
    status, nodes, _ = pp.kpath_matching(inst.bw_kbps, np.array([9, 7, 7, 3, 1], np.uint64), 2, draws)
    assert status == pp.PP_OK and len(set(nodes.tolist())) == 6
    seen["match"] = pp.debug_bounds_checks(MATCH)
    inst = W.config_resnet50_shaped()
    nseg, ends, nodes = W.random_plans(inst, 500, seed=2, invalid_fraction=0.2)
    off, e16, n8 = W.pack_plans(nseg, ends, nodes)
    draws = np.random.default_rng(6).integers(0, 2**32, size=(300, 2 * inst.k), dtype=np.uint64).astype(np.uint32)
    scored, drawn = oracle.eval_plans(inst, nseg, ends, nodes), OR.random_plans(inst, draws)
    with pp.Problem.from_instance(inst) as p:
        for name, got in (("eval", p.eval_plans(nseg, ends, nodes)), ("packed", p.eval_plans_packed(nseg, off, e16, n8))):
            assert np.array_equal(got[0], scored[0]) and np.array_equal(got[1], scored[1])
            seen[name] = pp.debug_bounds_checks(EVAL)
            p.eval_plans(nseg, ends, nodes)
        got = p.random_plans(draws)
        assert [a.tolist() for a in got] == list(drawn)
        seen["random"] = pp.debug_bounds_checks(RANDOM)
    return seen


def test_every_kernel_checks_its_tables():
    build.build()
    with library(build.build_debug()):
        seen = run_everything()
    assert all(n > 0 for n in seen.values()), seen
    assert set(run_everything().values()) == {0}
