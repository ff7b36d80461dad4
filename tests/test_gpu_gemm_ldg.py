"""bf16 products whose operands the CTA's threads stage themselves (rows off the 16-byte grid, long periods, narrow
pattern tiles) against the oracle: edges of the 128-row and 64 / 128-column tiles and of the 64-deep blocks, every
16-byte phase of a row, each cut of the contraction (1, 2, 4, 8 CTAs) and the form with 128-column tiles."""
import numpy as np
import pytest

from paper_2203_05705_b200 import ard, inputs
from gpu_helpers import Ctx, run_three_gemms, assert_ok, TOL

pytestmark = pytest.mark.gpu


def _layer(B, K, N, seed):
    rng = np.random.default_rng(seed)
    f = lambda *s: inputs.bf16_round(rng.standard_normal(s).astype(np.float32))  # noqa: E731
    return f(B, K), inputs.bf16_round((rng.standard_normal((K, N)) / np.sqrt(K)).astype(np.float32)), f(B, N)


@pytest.fixture(scope="module")
def ctx():
    c = Ctx(32 << 20)
    yield c
    c.close()


# K = 1001 .. 1006: rows start in every even 16-byte phase; 127 / 129, 63 / 65: tile and block edges; (20, 3000, 1500): an
# LSTM gate product; (700, 1500, 1500): 72 tiles cut in 4; (1500, 1300, 1900): 128-column tiles
@pytest.mark.parametrize("B,K,N", [(1, 17, 17), (127, 63, 129), (129, 65, 127), (130, 1001, 66), (64, 1002, 333), (20, 3000, 1500),
                                   (40, 1003, 90), (33, 1005, 1006), (700, 1500, 1500), (1500, 1300, 1900)])
def test_row_pattern_off_the_grid(ctx, B, K, N):
    X, W, dY = _layer(B, K, N, B + K + N)
    pat = ctx.pattern(ard.ARD_ROW, K, N)
    for i, (dp, b) in enumerate([(1, 1), (2, 2), (3, 1), (16, 7)]):
        if dp > N:
            continue
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        res = run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_BF16, X, W, dY, dp, b, 1.5, compact=(i % 2 == 1),
                              zero_fill=(i != 2), dw_dtype=ard.ARD_F32 if i % 2 else ard.ARD_BF16,
                              lds={"x": K + i, "w": K + 3 * (i & 1), "y": N + 5 * (i & 2)})
        assert_ok(res, TOL[ard.ARD_BF16], (B, K, N, dp, b))


@pytest.mark.parametrize("dp,b", [(40, 33), (100, 100)])
def test_row_pattern_with_a_long_period(ctx, dp, b):
    B, K, N = 150, 264, 1000
    X, W, dY = _layer(B, K, N, dp)
    pat = ctx.pattern(ard.ARD_ROW, K, N)
    ard.ard_pattern_set(ctx.h, pat, dp, b)
    assert_ok(run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_BF16, X, W, dY, dp, b, 2.0), TOL[ard.ARD_BF16], (dp, b))


@pytest.mark.parametrize("ts,B,Tr,Tc", [(32, 100, 3, 5), (32, 130, 64, 64), (32, 64, 7, 16), (16, 65, 9, 10), (8, 40, 20, 33),
                                        (32, 1300, 44, 48)])
def test_narrow_pattern_tiles(ctx, ts, B, Tr, Tc):
    K, N = Tr * ts, Tc * ts
    X, W, dY = _layer(B, K, N, ts + Tr)
    pat = ctx.pattern(ard.ARD_TILE, K, N, ts)
    for i, dp in enumerate([1, 2, 3, 5, 8, 15]):
        b = 1 + (3 * i) % dp
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        res = run_three_gemms(ctx, pat, ard.ARD_TILE, ard.ARD_BF16, X, W, dY, dp, b, 2.0, ts=ts, zero_fill=(i % 2 == 0),
                              dw_dtype=ard.ARD_F32 if i % 2 else ard.ARD_BF16)
        assert_ok(res, TOL[ard.ARD_BF16], (ts, B, Tr, Tc, dp, b))


@pytest.mark.parametrize("B,N", [(9475, 131), (2402, 131), (1187, 515)])
def test_compaction_of_tall_gradients(ctx, B, N):
    """The pass that compacts dY off the 16-byte grid takes 8, 4 or 1 rows per block: a last group that is not full."""
    rng = np.random.default_rng(B)
    K = 26
    X = inputs.bf16_round(rng.standard_normal((B, K)).astype(np.float32))
    W = inputs.bf16_round((rng.standard_normal((K, N)) * 0.05).astype(np.float32))
    dY = inputs.bf16_round(rng.standard_normal((B, N)).astype(np.float32))
    pat = ctx.pattern(ard.ARD_ROW, K, N)
    for dp, b in [(2, 2), (7, 3)]:
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        res = run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_BF16, X, W, dY, dp, b, 2.0)
        assert_ok(res, TOL[ard.ARD_BF16], (B, N, dp))
