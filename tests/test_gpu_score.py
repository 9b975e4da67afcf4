"""The plan evaluator where its staging can go wrong (batches around the block size, odd numbers of nodes,
rows far apart, unaligned arrays) and the random plans at odd sizes, against the oracles."""
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


@pytest.mark.parametrize("L,k,B", [(1, 1, 3), (2, 3, 255), (9, 5, 256), (30, 7, 257), (50, 14, 1000), (200, 18, 513), (1024, 20, 300)])
def test_rows_of_every_kind(L, k, B):
    import torch
    inst = W.random_small(93000 + L, L, k, dead_links=0.1)
    inst.node_mem_bytes[:] = np.uint64(int(inst.layer_mem_bytes.sum()) // 3 + 40_000_000)
    if L > 2:
        nseg, ends, nodes = W.random_plans(inst, B, seed=L, invalid_fraction=0.2)
    else:
        rng = np.random.default_rng(L)
        nseg = rng.integers(0, 4, B).astype(np.uint8)
        ends, nodes = rng.integers(-1, L + 1, (B, k)).astype(np.int32), rng.integers(-1, k + 1, (B, k)).astype(np.int32)
    want = oracle.eval_plans(inst, nseg, ends, nodes)
    off, e16, n8 = W.pack_plans(nseg, ends, nodes)
    with pp.Problem.from_instance(inst) as p:
        for got in (p.eval_plans(nseg, ends, nodes), p.eval_plans_packed(nseg, off, e16, n8)):
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        # rows with room to spare: a block's plans no longer fit its staging buffer
        keep = np.diff(off.astype(np.int64))
        wide = np.zeros(B + 1, np.uint32)
        wide[1:] = np.cumsum(keep + 3 * k)
        far_e, far_n = np.full(int(wide[-1]), 0xFFFF, np.uint16), np.full(int(wide[-1]), 0xFF, np.uint8)
        for b in range(B):
            far_e[wide[b]:wide[b] + keep[b]] = e16[off[b]:off[b + 1]]
            far_n[wide[b]:wide[b] + keep[b]] = n8[off[b]:off[b + 1]]
        got = p.eval_plans_packed(nseg, wide, far_e, far_n)
        ok = keep > 0  # a row without entries of its own now has some: flagged by them, if at all
        assert np.array_equal(got[0][ok], want[0][ok]) and np.array_equal(got[1][ok], want[1][ok])
        # arrays that start one entry into a buffer
        dev = [torch.from_numpy(a.view("i%d" % a.itemsize) if a.itemsize > 1 else a).cuda() for a in (
            np.concatenate([[0], nseg]).astype(np.uint8), off, np.concatenate([[0], e16]).astype(np.uint16),
            np.concatenate([[0], n8]).astype(np.uint8))]
        beta = torch.zeros(B, dtype=torch.float64, device="cuda")
        stat = torch.zeros(B, dtype=torch.uint8, device="cuda")
        p.eval_plans_packed_dev(B, e16.size, dev[0].data_ptr() + 1, dev[1].data_ptr(), dev[2].data_ptr() + 2,
                                dev[3].data_ptr() + 1, beta.data_ptr(), stat.data_ptr())
        assert np.array_equal(beta.cpu().numpy(), want[0]) and np.array_equal(stat.cpu().numpy(), want[1])


@pytest.mark.parametrize("L,k,P", [(1, 1, 5), (3, 2, 127), (40, 7, 129), (50, 20, 300), (1024, 13, 200)])
def test_random_plans_odd_shapes(L, k, P):
    inst = W.random_small(94000 + L, L, k)
    inst.node_mem_bytes[:] = (inst.node_mem_bytes.astype(np.float64) * max(1.0, L / (2.0 * k))).astype(np.uint64)
    draws = np.random.default_rng(k).integers(0, 2**32, size=(P, 2 * k), dtype=np.uint64).astype(np.uint32)
    with pp.Problem.from_instance(inst) as p:
        got = p.random_plans(draws)
    want = OR.random_plans(inst, draws)
    assert got[0].tolist() == want[0] and got[1].tolist() == want[1] and got[2].tolist() == want[2]
