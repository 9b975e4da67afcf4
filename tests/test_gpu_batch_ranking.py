"""The batched search's ranking of the quotients where its buckets can go wrong: quotients over the whole
range the limits allow, zero transfers, single values, and quotients equal to within the last bits."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W

pytestmark = pytest.mark.gpu


def extreme_instances(L, k, n=72):
    rng = np.random.default_rng(100 * L + k)
    insts = []
    for i in range(n):
        base = W.random_small(95000 + 100 * L + i, L, k)
        bits = base.layer_out_bits.copy()
        bw = rng.integers(1, 1 << 24, (k, k)).astype(np.uint32)
        kind = i % 6
        if kind == 0:    # the whole range of both, on a logarithmic scale
            bits = np.minimum(np.exp2(rng.uniform(0, 40, L)), (1 << 40) - 1).astype(np.uint64)
            bw = np.exp2(rng.uniform(0, 24, (k, k))).astype(np.uint32)
        elif kind == 1:  # transfers of nothing among others
            bits[rng.random(L) < 0.4] = 0
        elif kind == 2:  # nothing but zeros, or one value everywhere
            bits[:] = 0 if i % 12 == 2 else 12345
            bw[:] = 777
        elif kind == 3:  # quotients that differ in the last bits only, and by one tiny one
            bits = np.uint64((1 << 40) - 300) + rng.integers(0, 200, L).astype(np.uint64)
            bits[0] = 1
            bw = rng.integers((1 << 24) - 3, 1 << 24, (k, k)).astype(np.uint32)
        elif kind == 4:  # hardly any links
            bw[rng.random((k, k)) < 0.7] = 0
        np.fill_diagonal(bw, 0)
        insts.append(W.Instance(L, k, bits, base.layer_mem_bytes, base.node_mem_bytes, bw, f"ranking[{i}]"))
    return insts


@pytest.mark.parametrize("L,k", [(7, 3), (24, 8), (32, 8), (17, 5)])
def test_extreme_and_close_quotients(L, k):
    build.build()
    insts = extreme_instances(L, k)
    got = pp.solve_exact_batch(L, k, *(np.stack([getattr(i, f) for i in insts]) for f in (
        "layer_out_bits", "layer_mem_bytes", "node_mem_bytes", "bw_kbps")))
    for b, inst in enumerate(insts):
        want = oracle.dp_naive(inst)
        assert got.status[b] == want.status and got.plan(b) == want.plan(), (L, k, b)
        assert got.beta_ms[b] == want.beta_ms or np.isinf(want.beta_ms), (L, k, b)


@pytest.mark.parametrize("L,k", [(3, 2), (16, 5), (17, 4), (31, 6), (33, 6), (45, 7), (66, 5), (127, 4), (129, 4), (132, 3), (258, 3),
                                 (516, 2)])
def test_block_per_instance_shapes(L, k):
    """Rows of every number of positions a lane, whole and ragged ones, in the block-per-instance kernel."""
    build.build()
    n = 8 if L <= 66 else 3
    insts = []
    for i in range(n):
        base = W.random_small(97000 + 100 * L + i, L, k)
        scale = (1.2 + 0.3 * i) * float(base.layer_mem_bytes.sum()) / float(base.node_mem_bytes.sum())
        insts.append(W.Instance(L, k, base.layer_out_bits, base.layer_mem_bytes,
                                np.ceil(base.node_mem_bytes * scale).astype(np.uint64), base.bw_kbps, f"shape[{i}]"))
    got = pp.solve_exact_batch(L, k, *(np.stack([getattr(i, f) for i in insts]) for f in (
        "layer_out_bits", "layer_mem_bytes", "node_mem_bytes", "bw_kbps")))
    for b, inst in enumerate(insts):
        want = oracle.dp_naive(inst)
        assert got.status[b] == want.status and got.plan(b) == want.plan(), (L, k, b)
        assert got.beta_ms[b] == want.beta_ms or np.isinf(want.beta_ms), (L, k, b)


@pytest.mark.parametrize("B", [395, 396, 800])
def test_host_batch_in_pieces(B):
    """A host batch that is launched in pieces (two or more from 256 KB of inputs on) gives what small ones give."""
    build.build()
    L, k = 40, 4
    insts = [W.random_small(99000 + i % 97, L, k) for i in range(B)]
    cap = [np.ceil(i.node_mem_bytes * (1.4 * float(i.layer_mem_bytes.sum()) / float(i.node_mem_bytes.sum()))).astype(np.uint64)
           for i in insts]
    arrays = (np.stack([i.layer_out_bits for i in insts]), np.stack([i.layer_mem_bytes for i in insts]), np.stack(cap),
              np.stack([i.bw_kbps for i in insts]))
    got = pp.solve_exact_batch(L, k, *arrays)
    for b in range(0, B, 97):  # the instances repeat after 97
        n = min(97, B - b)
        part = pp.solve_exact_batch(L, k, *(a[:n] for a in arrays))
        for x, y in zip((got.beta_ms, got.m, got.cuts, got.placement, got.status),
                        (part.beta_ms, part.m, part.cuts, part.placement, part.status)):
            assert np.array_equal(x[b:b + n], y)
    assert (got.status == pp.PP_OK).any()
