"""Tile lists of the device sampler where a column's rows and the running counts can go wrong: more tile-columns than the sampler
has threads, periods longer than a column or than the grid of tiles is wide, periods that share factors with its width."""
import numpy as np
import pytest

from oracle import pattern as OP
from paper_2203_05705_b200 import ard
from gpu_helpers import Ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Tr,Tc", [(1, 1), (3, 1025), (2, 2500), (70, 12), (33, 31), (1, 40), (64, 64)])
def test_every_kind_of_period(Tr, Tc):
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_TILE, Tr, Tc, 1)
        units = Tr * Tc
        for dp in sorted({d for d in (1, 2, 3, 4, 5, 6, 12, 31, 62, 64, Tr + 1, Tc - 1, Tc, Tc + 1, 2 * Tc, units - 1, units) if 1 <= d <= units}):
            for b in sorted({1, (dp + 1) // 2, dp}):
                ard.ard_pattern_set(ctx.h, pat, dp, b)
                got = ard.ard_pattern_tile_lists_to_host(pat, Tr, Tc)
                for g, o in zip(got, OP.tile_lists(Tr, Tc, 1, dp, b)):
                    assert np.array_equal(g, o), (Tr, Tc, dp, b)
    finally:
        ctx.close()


@pytest.mark.parametrize("dp,b", [(2 ** 26, 1), (2 ** 26 + 1, 6), (2 ** 25, 1)])
def test_rows_whose_distance_times_a_warp_is_no_int(dp, b):
    Tr = 2 ** 26 + 1
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_TILE, Tr, 1, 1)
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        col_ptr, col_idx, row_ptr, row_idx = ard.ard_pattern_tile_lists_to_host(pat, Tr, 1)
        rows = np.arange(b - 1, Tr, dp)
        assert np.array_equal(col_ptr, [0, len(rows)]) and np.array_equal(col_idx[:len(rows)], rows)
        assert row_ptr[-1] == len(rows) and not row_idx[:len(rows)].any()
    finally:
        ctx.close()
