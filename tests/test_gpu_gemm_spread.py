"""Layers off the 16-byte grid that are wide and shallow, under long periods: a full-width output or a weight gradient is then
many times as large as the product behind it, and its zeros are dealt to more CTAs than the product has tiles.  Contractions
of one to three blocks (not cut) and longer ones, rows at every phase of the grid, both output types, few and many rows."""
import numpy as np
import pytest

from paper_2203_05705_b200 import ard, inputs
from gpu_helpers import Ctx, run_three_gemms, assert_ok, TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [ard.ARD_BF16, ard.ARD_F32])
@pytest.mark.parametrize("B,K,N", [(129, 130, 2047), (1000, 70, 2045), (20, 300, 4001), (17, 131, 1998), (2000, 129, 517), (1, 33, 3003)])
def test_zeros_of_wide_layers(dtype, B, K, N):
    rng = np.random.default_rng(B + N)
    r = inputs.bf16_round if dtype == ard.ARD_BF16 else (lambda a: a)
    X, dY = (r(rng.standard_normal(s).astype(np.float32)) for s in ((B, K), (B, N)))
    W = r((rng.standard_normal((K, N)) / np.sqrt(K)).astype(np.float32))
    ctx = Ctx(2 * B * (N + 8) + 4096)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        for i, (dp, b) in enumerate([(16, 16), (7, 1), (16, 5), (2, 2)]):
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_ROW, dtype, X, W, dY, dp, b, 1.5, zero_fill=True,
                                  dw_dtype=ard.ARD_F32 if i % 2 else dtype, lds={"x": K + i, "w": K + 3 * i, "y": N + i})
            assert_ok(res, TOL[dtype], (B, K, N, dp, b))
    finally:
        ctx.close()


# 192- and 256-wide bf16 tiles with aligned rows: the tensor-core kernels of a fixed tile width; others off the grid now and then
@pytest.mark.parametrize("dtype,ts,Tr,Tc", [(ard.ARD_F32, 256, 3, 4), (ard.ARD_F32, 96, 7, 5), (ard.ARD_BF16, 32, 40, 33), (ard.ARD_F32, 5, 9, 11),
                                            (ard.ARD_BF16, 256, 4, 3), (ard.ARD_BF16, 192, 3, 5)])
def test_zeros_of_tiles_of_every_size(dtype, ts, Tr, Tc):
    B, K, N = 9, Tr * ts, Tc * ts
    rng = np.random.default_rng(ts)
    r = inputs.bf16_round if dtype == ard.ARD_BF16 else (lambda a: a)
    X, dY = (r(rng.standard_normal(s).astype(np.float32)) for s in ((B, K), (B, N)))
    W = r((rng.standard_normal((K, N)) / np.sqrt(K)).astype(np.float32))
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_TILE, K, N, ts)
        for i, (dp, b) in enumerate([(2, 1), (5, 5), (11, 4)]):
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            for dw in {dtype, ard.ARD_F32}:
                res = run_three_gemms(ctx, pat, ard.ARD_TILE, dtype, X, W, dY, dp, b, 2.0, ts=ts, dw_dtype=dw,
                                      lds={"w": K + 8 * (i % 2) + (i == 2)})
                assert_ok(res, TOL[dtype], (ts, dp, b))
    finally:
        ctx.close()
