"""Recurrences inside clusters of CTAs, forward and backward against the oracle, at the edges of the kernels: most units of a
cluster of 8 and of 16 CTAs and one more, one unit, a second and a third group of 8 batch rows, the three ways the weights come in
(periods of 1 and 2 with rows on the 8 and 16 byte grid, from every phase of it, and everything else), weight-gradient rows longer than what a copy of
zeros holds, and more steps than one burst of them.  What the weights of dropped
units hold does not matter."""
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


@pytest.mark.parametrize("T,B,I,H,dp,b", [
    (3, 121, 16, 384, 1, 1), (3, 16, 20, 385, 1, 1), (3, 113, 40, 768, 1, 1), (2, 20, 40, 769, 1, 1), (3, 9, 8, 1536, 2, 2),
    (2, 60, 24, 1538, 2, 1), (3, 57, 52, 1504, 2, 2), (2, 5, 37, 769, 2, 2), (4, 1, 16, 17, 1, 1), (3, 2, 64, 12, 12, 7),
    (3, 8, 50, 122, 1, 1), (3, 8, 51, 121, 1, 1), (3, 64, 30, 506, 2, 1), (3, 64, 30, 506, 2, 2), (1, 30, 44, 260, 3, 3),
    (3, 128, 24, 1024, 2, 1), (5, 64, 64, 400, 16, 16),
    (3, 57, 24, 1024, 2, 1), (3, 120, 40, 1023, 2, 2), (2, 120, 16, 385, 1, 1), (18, 9, 4104, 120, 4, 3)])
def test_edges_of_the_cluster_recurrences(T, B, I, H, dp, b):
    rng = np.random.default_rng(T * 1000 + B + H)
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(I + H, 4 * H)).astype(np.float32))
    X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
    dH = (rng.standard_normal((T, B, H)) / 8).astype(np.float32)
    m, keep = OP.row_mask(H, dp, b), OP.row_keep(H, dp, b)
    fw = OL.fwd(X, W, None, m, 1.5)
    bw = OL.bwd(fw, W, m, 1.5, dH)
    Wd = W.copy()
    drop = np.where(m == 0)[0]
    Wd[I + drop, :] = np.nan
    for g in range(4):
        Wd[:, g * H + drop] = np.nan
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, T, B, I, H, torch.from_numpy(np.ascontiguousarray(Wd.T)).to(BF).cuda())
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        layer.XH[1:, :, I:] = float("nan")
        for buf in (layer.D, layer.dc, layer.dW, layer.G):
            buf.fill_(float("nan"))
        layer.load_inputs(torch.from_numpy(X).to(BF).cuda())
        h = layer.forward(1.5)
        dX, dW = layer.backward(1.5, torch.from_numpy(dH).cuda())
        assert ard.ard_last_device_status(ctx.h) == 0
        n = len(keep)
        assert OG.rel_fro(host(h.float()), fw["Hs"]) <= TOL[ard.ARD_BF16]
        assert bool(torch.all(h[:, :, torch.from_numpy(m == 0).cuda()] == 0))
        assert OG.rel_fro(host(layer.C[T, :, :n]), fw["cT"][:, keep]) <= TOL[ard.ARD_BF16]
        assert OG.rel_fro(host(dX), bw["dX"]) <= TOL[ard.ARD_BF16]
        assert OG.rel_fro(host(dW), bw["dW"].T) <= TOL[ard.ARD_BF16]
        assert OG.rel_fro(host(layer.D[0, :, I:]), bw["dh0"] * m[None, :]) <= TOL[ard.ARD_BF16]
        assert OG.rel_fro(host(layer.dc[:, :n]), bw["dc0"][:, keep]) <= TOL[ard.ARD_BF16]
        assert bool((layer.dc[:, n:] == 0).all())
    finally:
        ctx.close()
