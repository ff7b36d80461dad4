"""Zeros of the dropped tiles of dW, written by the weight gradient of the class form: both output types and tile sizes,
first / middle / last kept tile of a period, more dropped tiles than there are warps writing them, a padded pitch."""
import numpy as np
import pytest

from paper_2203_05705_b200 import ard, inputs
from gpu_helpers import Ctx, run_three_gemms, assert_ok, TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ts,rows,cols,dw", [(64, 44, 32, ard.ARD_BF16), (64, 3, 5, ard.ARD_F32), (128, 5, 3, ard.ARD_F32),
                                             (128, 4, 4, ard.ARD_BF16)])
def test_dropped_tiles_are_zero(ts, rows, cols, dw):
    B, K, N = 24, rows * ts, cols * ts
    rng = np.random.default_rng(ts + rows)
    X = inputs.bf16_round(rng.standard_normal((B, K)).astype(np.float32))
    W = inputs.bf16_round((rng.standard_normal((K, N)) * 0.05).astype(np.float32))
    dY = inputs.bf16_round(rng.standard_normal((B, N)).astype(np.float32))
    ctx = Ctx(1 << 20)
    try:
        ard.ard_set_path(ctx.h, ard.ARD_PATH_TENSOR_CORE)
        pat = ctx.pattern(ard.ARD_TILE, K, N, ts)
        for i, (dp, b) in enumerate([(2, 1), (2, 2), (3, 2), (7, 7), (rows * cols, rows * cols // 2)]):
            if dp > 64:
                continue
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_TILE, ard.ARD_BF16, X, W, dY, dp, b, 2.0, ts=ts, zero_fill=True, dw_dtype=dw,
                                  lds={"w": K + 8 * (i % 2)})
            assert_ok(res, TOL[ard.ARD_BF16], (ts, dp, b))
    finally:
        ctx.close()
