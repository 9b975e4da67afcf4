"""Which batches go an instance to a lane, which to a warp, which to blocks of 192 threads and which to blocks of 384, by the library's own rule
(no device is needed).  Every line was measured on both sides; the times stand beside the rules."""
from __future__ import annotations

import pytest

import paper_2210_12219_b200 as pp
from paper_2210_12219_b200 import build

LANES, WARPS, NARROW, WIDE = 0, 32, 192, 384


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("L,k,held", [(45, 6, 6), (66, 6, 5), (80, 6, 4), (91, 6, 3), (125, 6, 2), (193, 6, 1), (80, 5, 6), (100, 5, 5),
                                      (125, 5, 4), (140, 5, 3), (180, 5, 2), (125, 4, 6), (160, 4, 4), (200, 4, 3), (256, 3, 5),
                                      (256, 2, 6), (257, 2, 0), (45, 7, 0)])
def test_narrow_blocks_take_fewer_waves(L, k, held):
    # held: narrow blocks an SM has room for; three wide ones, or as many as narrow ones where that is fewer
    for B in (1, 64, 444, 445, 500, 592, 593, 740, 888, 889, 900, 1184, 1185, 1332, 1500, 1776, 1777, 2221, 4000, 100_000):
        waves = lambda blocks: -(-B // (148 * blocks))
        if held == 0:
            want = False
        elif held > 4 or k == 4:
            want = waves(held) < waves(3)
        else:
            want = 3 * waves(held) <= 2 * waves(min(held, 3))
        assert pp.debug_batch_route(B, L, k) == (NARROW if want else WIDE), B


@pytest.mark.parametrize("L,k,B,want", [(20, 6, 600, NARROW), (24, 6, 1000, NARROW), (32, 4, 1000, NARROW), (33, 6, 600, WIDE), (40, 5, 1000, WIDE),
                                        (33, 6, 500, NARROW), (33, 6, 740, WIDE), (33, 6, 1000, NARROW), (36, 6, 1100, NARROW), (37, 6, 1000, WIDE),
                                        (60, 6, 740, WIDE), (100, 6, 560, WIDE), (33, 6, 100, WIDE), (60, 6, 2000, NARROW),
                                        (60, 7, 800, WIDE)])
def test_host_batches_count_a_piece_of_long_chains(L, k, B, want):
    # up to 1 MB a host batch goes in pieces, of which two count up to 36 layers and one beyond; 2000 x (60, 6) is more
    # and goes as a device batch does
    assert pp.debug_batch_route(B, L, k, host=True) == want
    if L > 32 and k <= 6:
        assert pp.debug_batch_route(B, L, k) == (NARROW if B > 444 and L < 91 else WIDE)


# batches of short chains: a wave of blocks (three to an SM, six narrow ones for k <= 6, two for k = 8 from 29 layers on), two waves, or
# one and a half go an instance to a block, larger ones an instance to a lane or a warp; host batches of up to 1 MB never do
@pytest.mark.parametrize("L,k,most", [(24, 2, 888), (16, 3, 888), (9, 4, 1776), (32, 4, 1776), (20, 5, 1776), (16, 6, 1776), (17, 6, 1332), (24, 6, 1332),
                                      (25, 6, 1776), (32, 6, 1776), (16, 7, 888), (17, 7, 444), (24, 7, 444), (25, 7, 888), (32, 7, 888),
                                      (16, 8, 888), (17, 8, 444), (28, 8, 444), (29, 8, 296), (32, 8, 296)])
def test_larger_batches_of_short_chains_share_blocks(L, k, most):
    for B in (1, 64, most):
        assert pp.debug_batch_route(B, L, k) in (NARROW, WIDE), B
    for B in (most + 1, 2 * most, 4096, 100_000):
        assert pp.debug_batch_route(B, L, k) in (LANES, WARPS), B
        assert pp.debug_batch_route(B, L, k) == LANES or k >= 6, B
        arrays = (8 * L, 8 * L, 8 * k, 4 * k * k, 8, 4, 4 * (k - 1), 4 * k, 1)  # bytes an instance
        in_place = sum(-(-B * a // 256) * 256 for a in arrays) <= 1 << 20
        assert (pp.debug_batch_route(B, L, k, host=True) in (NARROW, WIDE)) == in_place, B


# the smallest batch of a shape that goes an instance to a warp; one that is smaller by one goes to a lane, or to a block where
# that is as far as the blocks go
@pytest.mark.parametrize("L,k,B", [(1, 8, 889), (9, 8, 889), (10, 8, 1500), (14, 8, 1500), (15, 8, 1800), (16, 8, 1800), (17, 8, 2000), (24, 8, 2000),
                                   (25, 8, 1500), (32, 8, 1500), (1, 7, 889), (6, 7, 889), (7, 7, 1700), (12, 7, 1700), (13, 7, 2100), (20, 7, 2100),
                                   (21, 7, 2500), (24, 7, 2500), (25, 7, 2000), (32, 7, 2000), (1, 6, 1777), (6, 6, 1777), (7, 6, 4097),
                                   (32, 6, 4097)])
def test_batches_an_instance_to_a_warp(L, k, B):
    for n in (B, B + 1, 2 * B, 100_000):
        assert pp.debug_batch_route(n, L, k) == WARPS, n
    assert pp.debug_batch_route(B - 1, L, k) in ((NARROW, WIDE) if B in (889, 1777) else (LANES,))


def test_the_lanes_are_asked_for_no_level_that_is_not_there():
    # rows of four words have the levels of seven nodes and fewer (kLanesShortK)
    for L in range(1, 9):
        for B in (*range(1, 2200, 7), *range(2200, 9000, 97), 4095, 4096, 4097, 100_000):
            assert pp.debug_batch_route(B, L, 8) != LANES, (B, L)


@pytest.mark.parametrize("L,k", [(33, 8), (24, 9), (24, 1)])
def test_other_shapes_never_do(L, k):
    for B in (1, 4096, 100_000):
        assert pp.debug_batch_route(B, L, k) in (NARROW, WIDE)
