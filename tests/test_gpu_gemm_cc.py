"""CUDA-core products against the oracle where their tiling can go wrong: edges of the 32- and 64-wide tiles and of the
contraction blocks, rows on and off the four-element grid, each cut of the contraction, pattern tiles of any size."""
import numpy as np
import pytest

from paper_2203_05705_b200 import ard, inputs
from gpu_helpers import Ctx, run_three_gemms, assert_ok, TOL

pytestmark = pytest.mark.gpu


def _layer(B, K, N, seed, bf16=False):
    rng = np.random.default_rng(seed)
    a = [rng.standard_normal(s).astype(np.float32) for s in ((B, K), (K, N), (B, N))]
    a[1] /= np.float32(np.sqrt(K))
    return [inputs.bf16_round(x) for x in a] if bf16 else a


@pytest.fixture(scope="module")
def ctx():
    c = Ctx(8 << 20)
    yield c
    c.close()


# 2 B K N below and above 2e8 picks 32- and 64-wide tiles
@pytest.mark.parametrize("B,K,N", [(31, 33, 65), (64, 784, 256), (33, 127, 31), (128, 2048, 2048), (65, 1601, 1003), (1030, 513, 400)])
def test_row_pattern(ctx, B, K, N):
    X, W, dY = _layer(B, K, N, B + K + N)
    pat = ctx.pattern(ard.ARD_ROW, K, N)
    ard.ard_set_path(ctx.h, ard.ARD_PATH_CUDA_CORE)
    try:
        for i, (dp, b) in enumerate([(1, 1), (2, 2), (3, 1), (16, 7)]):
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_F32, X, W, dY, dp, b, 1.5, compact=(i % 2 == 1), zero_fill=(i != 2),
                                  lds={"x": K + i, "w": K + 3 * (i & 1), "y": N + 5 * (i & 2)})
            assert_ok(res, TOL[ard.ARD_F32], (B, K, N, dp, b))
    finally:
        ard.ard_set_path(ctx.h, ard.ARD_PATH_AUTO)


@pytest.mark.parametrize("dtype", [ard.ARD_F32, ard.ARD_BF16])
@pytest.mark.parametrize("ts,B,Tr,Tc", [(32, 100, 3, 5), (64, 130, 32, 32), (5, 40, 20, 33), (12, 65, 9, 10), (128, 70, 6, 7), (1, 20, 40, 50)])
def test_tile_pattern(ctx, dtype, ts, B, Tr, Tc):
    K, N = Tr * ts, Tc * ts
    X, W, dY = _layer(B, K, N, ts + Tr, dtype == ard.ARD_BF16)
    pat = ctx.pattern(ard.ARD_TILE, K, N, ts)
    ard.ard_set_path(ctx.h, ard.ARD_PATH_CUDA_CORE)
    try:
        for i, dp in enumerate([1, 2, 3, 5, 8, 15]):
            b = 1 + (3 * i) % dp
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_TILE, dtype, X, W, dY, dp, b, 2.0, ts=ts, zero_fill=(i % 2 == 0))
            assert_ok(res, TOL[dtype], (ts, B, Tr, Tc, dp, b))
    finally:
        ard.ard_set_path(ctx.h, ard.ARD_PATH_AUTO)
