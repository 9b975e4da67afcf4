"""A search whose blocks wait for one that never comes gives up after a bounded number of polls: it reports that on
every path, and leaves the counters clean for the search after it."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build
from paper_2210_12219_b200 import workloads as W
from tests.test_gpu_errors import library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    pp.lib()


def record(sol):
    import torch
    torch.cuda.synchronize()
    return pp.pp_solution.from_buffer_copy(sol.cpu().numpy().tobytes()[:176])


@pytest.mark.parametrize("inst", [W.config_resnet50_shaped(), W.config_deeper_cnn(), W.config_geometric(13, 64, 3)],
                         ids=lambda i: f"k{i.k}")
def test_search_reports_a_wait_that_ran_out(inst):
    import torch
    want = oracle.dp_fact(inst, 8)
    sol = torch.zeros(22, dtype=torch.float64, device="cuda")
    with pp.Problem.from_instance(inst) as p:
        p.set_stream(torch.cuda.current_stream().cuda_stream)
        for polls in (1, 3000):  # 3000: past the point where the blocks ask whether another one has given up
            p.solve_exact_dev(sol.data_ptr())  # a sound record first, which must not be taken for the next one
            assert record(sol).status == pp.PP_OK
            pp.debug_starve(polls)
            p.solve_exact_dev(sol.data_ptr())
            got = record(sol)
            assert (got.status, got.m, got.beta_ms) == (pp.PP_ERR_CUDA, 0, np.inf)
            assert list(got.placement) == [-1] * pp.PP_MAX_K
            for _ in range(3):  # the counters were cleared: blocks that did not wait would show up here
                p.solve_exact_dev(sol.data_ptr())
                got = record(sol)
                assert got.status == pp.PP_OK and got.beta_ms == want.beta_ms
                assert (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == want.plan()
        pp.debug_starve(50)
        with pytest.raises(pp.PPError) as e:
            p.solve_exact()
        assert e.value.status == pp.PP_ERR_CUDA
        got = p.solve_exact()
        assert got.beta_ms == want.beta_ms and got.plan() == want.plan()


def test_eq1_and_placement_report_a_wait_that_ran_out():
    inst = W.config_geometric(12, 64, 1)
    work = (inst.layer_mem_bytes // np.uint64(1024)).astype(np.uint64)
    speed = (1000 + 37 * np.arange(inst.k)).astype(np.uint32)
    first = pp.solve_exact_compute(inst, work, speed)
    pp.debug_starve(50)
    with pytest.raises(pp.PPError) as e:
        pp.solve_exact_compute(inst, work, speed)
    assert e.value.status == pp.PP_ERR_CUDA
    again = pp.solve_exact_compute(inst, work, speed)
    assert again.beta_ms == first.beta_ms and again.plan() == first.plan()

    draws = np.random.default_rng(5).integers(0, 2**32, size=(12, inst.k), dtype=np.uint64).astype(np.uint32)
    sizes = np.array([9, 7, 7, 3, 1], np.uint64)
    first = pp.kpath_matching(inst.bw_kbps, sizes, 2, draws)
    pp.debug_starve(50)
    with pytest.raises(pp.PPError) as e:
        pp.kpath_matching(inst.bw_kbps, sizes, 2, draws)
    assert e.value.status == pp.PP_ERR_CUDA
    for _ in range(3):  # both halves of the records
        again = pp.kpath_matching(inst.bw_kbps, sizes, 2, draws)
        assert again[0] == first[0] and np.array_equal(again[1], first[1]) and np.array_equal(again[2], first[2])
    pp.debug_starve(0)


def test_a_block_that_comes_late_to_the_vote_gives_up_with_the_others():
    """Blocks that decide a threshold each: one of them, whichever it is, comes to the last vote when the others have given up.
    All give up then, and the error is on record; the late one does not go on alone with what the others were to write."""
    import torch
    inst = W.config_geometric(8, 48, 2)
    want = oracle.dp_fact(inst, 8)
    work = (inst.layer_mem_bytes // np.uint64(1024)).astype(np.uint64)
    speed = (1000 + 37 * np.arange(inst.k)).astype(np.uint32)
    sol = torch.zeros(22, dtype=torch.float64, device="cuda")
    with library(build.build_debug()):
        first = pp.solve_exact_compute(inst, work, speed)
        with pp.Problem.from_instance(inst) as p:
            for late in range(torch.cuda.get_device_properties(0).multi_processor_count):
                p.solve_exact_dev(sol.data_ptr())  # a sound record first, which must not be taken for the next one
                assert record(sol).status == pp.PP_OK
                pp.debug_late(late, 3000)
                p.solve_exact_dev(sol.data_ptr())
                got = record(sol)
                assert (got.status, got.m, got.beta_ms) == (pp.PP_ERR_CUDA, 0, np.inf), late
                assert list(got.placement) == [-1] * pp.PP_MAX_K
                p.solve_exact_dev(sol.data_ptr())
                got = record(sol)
                assert got.status == pp.PP_OK and got.beta_ms == want.beta_ms
                assert (got.m, tuple(got.cuts[: got.m - 1]), tuple(got.placement[: got.m])) == want.plan()
                pp.debug_late(late, 3000)
                with pytest.raises(pp.PPError) as e:
                    pp.solve_exact_compute(inst, work, speed)
                assert e.value.status == pp.PP_ERR_CUDA, late
        again = pp.solve_exact_compute(inst, work, speed)
        assert again.beta_ms == first.beta_ms and again.plan() == first.plan()
    with pytest.raises(pp.PPError):
        pp.debug_late(0, 1)  # the normal build has no such hook
