"""The one-launch placement stage at its edges (more colourings than blocks, the longest run it takes and
the first one it leaves to the bisection), and the partition stage's queue on windows of every kind,
against the oracles."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2210_12219_b200 as pp
from oracle import partition as OP
from oracle import placement as OPL
from paper_2210_12219_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    pp.lib()


@pytest.mark.parametrize("n,cuts,classes,trials", [(12, 5, 2, 200), (13, 8, 1, 60), (14, 9, 1, 40), (64, 4, 2, 10), (2, 1, 1, 3),
                                                   (13, 11, 1, 30), (32, 5, 2, 9), (33, 5, 2, 9), (3, 2, 1, 149)])
def test_matching_shapes(n, cuts, classes, trials):
    rng = np.random.default_rng(n * 100 + cuts)
    for sym in (True, False):
        bw = rng.integers(0, 60, size=(n, n)).astype(np.uint32)
        if sym:
            bw = (np.triu(bw, 1) + np.triu(bw, 1).T).astype(np.uint32)
        sizes = rng.integers(1, 9, cuts).astype(np.uint64)
        draws = rng.integers(0, 2**32, size=(trials, n), dtype=np.uint64).astype(np.uint32)
        want = OPL.k_path_matching(bw.tolist(), [int(x) for x in sizes], classes, draws.tolist())
        st, nodes, thr = pp.kpath_matching(bw, sizes, classes, draws)
        if want.status == OPL.INFEASIBLE:
            assert st == pp.PP_INFEASIBLE and (nodes == -1).all()
            continue
        assert st == pp.PP_OK and tuple(nodes.tolist()) == want.nodes
        for first, run, _, t in want.thresholds:
            assert (thr[first:first + run] == t).all()


@pytest.mark.parametrize("L", [1, 2, 31, 32, 33, 64, 65, 100, 128, 129, 1024])
def test_partition_windows(L):
    # windows from a single point to the whole chain, equal and rising and falling weights
    rng = np.random.default_rng(L)
    weights = [rng.integers(1, 1000, L), np.full(L, 7), np.arange(1, L + 1), np.arange(L, 0, -1)]
    mem = [rng.integers(1, 10, L), np.ones(L, int)]
    for w in weights:
        for m in mem:
            for kappa in (int(m.max()), int(m.max()) + 1, int(m.sum()) // 3 + 9, int(m.sum())):
                want = OP.minsum_partition([int(x) for x in w], [int(x) for x in m], kappa) if L <= 129 else None
                got = pp.partition_minsum_batch(w[None].astype(np.uint64), m[None].astype(np.uint64),
                                                np.array([kappa], np.uint64), L)
                many = pp.partition_minsum_batch(np.repeat(w[None], 40, 0).astype(np.uint64),
                                                 np.repeat(m[None], 40, 0).astype(np.uint64), np.full(40, kappa, np.uint64), L)
                assert (many.cost == got.cost[0]).all() and (many.cuts == got.cuts[0]).all() and got.status[0] == pp.PP_OK
                if want is None:  # the plan is consistent: it costs what it says and every part fits
                    parts = int(got.m[0])
                    cut = got.cuts[0, :parts - 1].tolist()
                    assert int(got.cost[0]) == int(sum(int(w[c]) for c in cut))
                    ends = [-1] + cut + [L - 1]
                    assert all(int(m[a + 1:b + 1].sum()) <= kappa for a, b in zip(ends, ends[1:]))
                else:
                    assert int(got.m[0]) == want.m and tuple(got.cuts[0, :want.m - 1].tolist()) == want.cuts
                    assert int(got.cost[0]) == int(sum(int(w[c]) for c in want.cuts))
