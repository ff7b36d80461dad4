"""Gate functions near zero: the whole-sequence kernels save tanh gates and cell states whose relative error is that of
fp32 sums and functions, whatever the layer's alignment, and hand back what the per-step kernels hand back."""
import numpy as np
import pytest
import torch

from oracle import pattern as OP
from paper_2203_05705_b200 import ard, inputs
from paper_2203_05705_b200.lstm import LstmLayer
from gpu_helpers import Ctx, host

pytestmark = pytest.mark.gpu
BF = torch.bfloat16
# x . W over I <= 64 products, each exact in fp32, added in any order: at most I * 2^-24 of the sum of magnitudes, which is
# about sqrt(I) times the sum: 64 * 8 * 6e-8 = 3e-5 at worst, about sqrt(I) * 2^-24 * 1.25 = 6e-7 for random signs; functions
# and products add a few 2^-24.  A quotient that cancels near zero is off by 2^-24 / 0.01 = 6e-6 at this input size.
RTOL = 2e-6


@pytest.mark.parametrize("B,I,H", [(20, 64, 128), (20, 52, 204), (33, 57, 131), (8, 64, 98), (70, 60, 1196)])
def test_small_gates_keep_their_relative_error(B, I, H):
    rng = np.random.default_rng(B + H)
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(I + H, 4 * H)).astype(np.float32))
    X = inputs.bf16_round((rng.standard_normal((1, B, I)) * 0.02).astype(np.float32))
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, 1, B, I, H, torch.from_numpy(np.ascontiguousarray(W.T)).to(BF).cuda())
        for dp, b in [(1, 1), (3, 2)]:
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            keep = OP.row_keep(H, dp, b)
            z = (X[0].astype(np.float64) @ W[:I].astype(np.float64)).reshape(B, 4, H)[:, :, keep]
            s = lambda v: 1.0 / (1.0 + np.exp(-v))  # noqa: E731
            g, c = np.tanh(z[:, 2]), s(z[:, 0]) * np.tanh(z[:, 2])
            layer.load_inputs(torch.from_numpy(X).to(BF).cuda())
            layer.forward(1.5)
            assert ard.ard_last_device_status(ctx.h) == 0
            G = host(layer.G).reshape(B, 4, H)[:, :, :len(keep)]
            C = host(layer.C[1])[:, :len(keep)]
            assert 1e-3 < np.abs(g).mean() < 2e-2       # where the relative error of a cancelling form shows
            assert np.linalg.norm(G[:, 2] - g) <= RTOL * np.linalg.norm(g), (dp, b)
            assert np.linalg.norm(C - c) <= RTOL * np.linalg.norm(c), (dp, b)
    finally:
        ctx.close()
