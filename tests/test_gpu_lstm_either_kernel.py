"""LSTM layers whose distribution has periods on both sides of what the clusters hold (768 units on 148 SMs): two kernels are enqueued per
recurrence and the drawn pattern decides which one works.  One, two and three groups of 8 rows in a cluster, a pattern of 768 units and one of
769, the most and the fewest units."""
import numpy as np
import pytest
import torch

from oracle import gemm as OG
from oracle import lstm as OL
from oracle import pattern as OP
from paper_2203_05705_b200 import ard, inputs
from paper_2203_05705_b200.lstm import LstmLayer
from gpu_helpers import Ctx, host, TOL

pytestmark = pytest.mark.gpu
BF = torch.bfloat16


@pytest.mark.parametrize("T,B,I,H", [(3, 9, 40, 1024), (2, 64, 24, 1023), (2, 128, 16, 1024), (2, 20, 24, 1536), (3, 20, 20, 1538)])
def test_the_drawn_pattern_decides(T, B, I, H):
    K = [0.3, 0.4] + [0.0] * 13 + [0.3]
    cdf = OP.quantise_K(K)
    rng = np.random.default_rng(H + B)
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(I + H, 4 * H)).astype(np.float32))
    X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
    dH = (rng.standard_normal((T, B, H)) / 8).astype(np.float32)
    ctx = Ctx(1 << 20)
    try:
        ard.ard_set_distribution(ctx.h, 0, K)
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, T, B, I, H, torch.from_numpy(np.ascontiguousarray(W.T)).to(BF).cuda())
        layer.load_inputs(torch.from_numpy(X).to(BF).cuda())
        dHd = torch.from_numpy(dH).cuda()
        for want in (2, 1, 16):
            it = next(i for i in range(1000) if OP.draw(cdf, 9, i, 0)[0] == want)
            dp, b = OP.draw(cdf, 9, it, 0)
            m, keep = OP.row_mask(H, dp, b), OP.row_keep(H, dp, b)
            ard.ard_sample_pattern(ctx.h, pat, 0, 9, it, 0)
            layer.XH[1:, :, I:] = float("nan")
            for buf in (layer.D, layer.dc, layer.dW, layer.G):
                buf.fill_(float("nan"))
            h = layer.forward(1.5)
            dX, dW = layer.backward(1.5, dHd)
            assert ard.ard_last_device_status(ctx.h) == 0
            fw = OL.fwd(X, W, None, m, 1.5)
            bw = OL.bwd(fw, W, m, 1.5, dH)
            tol = TOL[ard.ARD_BF16]
            assert OG.rel_fro(host(h.float()), fw["Hs"]) <= tol, dp
            assert OG.rel_fro(host(dX), bw["dX"]) <= tol, dp
            assert OG.rel_fro(host(dW), bw["dW"].T) <= tol, dp
            assert OG.rel_fro(host(layer.D[0, :, I:]), bw["dh0"] * m[None, :]) <= tol, dp
            assert OG.rel_fro(host(layer.dc[:, :len(keep)]), bw["dc0"][:, keep]) <= tol, dp
    finally:
        ctx.close()
