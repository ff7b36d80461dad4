"""Whole-sequence LSTM kernels on layers off the 16-byte grid and of more than 8 units per SM, forward and backward against
the oracle: gate blocks, h columns and rows at every phase, a ring of slots that is re-used within a step, 4, 8 and 12 units
per CTA, shared and whole contractions of the gradients (clusters of CTAs with units for some of them only, a layer whose
CTAs do not fit the device in clusters), one and two row boxes; and a layer whose backward pass does not fit and runs step by step."""
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


# (KH % 8 == 0, H % 8 == 4), odd everything, H % 4 == 2, > 1024 units at one and two row boxes, > 1184 units (12 per CTA),
# does not fit; few CTAs, not a multiple of a cluster, two CTAs, more CTAs than clusters of them fit
@pytest.mark.parametrize("T,B,I,H,fits", [(4, 20, 52, 204, 1), (3, 33, 57, 131, 1), (3, 8, 64, 98, 1), (3, 70, 36, 1100, 1),
                                          (3, 128, 64, 1096, 1), (3, 20, 300, 1500, 1), (2, 100, 44, 1500, 0),
                                          (4, 9, 24, 40, 1), (3, 40, 24, 604, 1), (3, 5, 16, 12, 1), (2, 8, 40, 1600, 1)])
def test_any_shape_matches_the_oracle(T, B, I, H, fits):
    rng = np.random.default_rng(T * 100 + B + H)
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(I + H, 4 * H)).astype(np.float32))
    X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
    dH = (rng.standard_normal((T, B, H)) / 8).astype(np.float32)
    Wnm = torch.from_numpy(np.ascontiguousarray(W.T)).to(BF).cuda()
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, T, B, I, H, Wnm)
        for dp, b in [(1, 1), (2, 2), (3, 1), (9, 5)]:
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            m, keep = OP.row_mask(H, dp, b), OP.row_keep(H, dp, b)
            fw = OL.fwd(X, W, None, m, 1.5)
            bw = OL.bwd(fw, W, m, 1.5, dH)
            layer.XH[1:, :, I:] = float("nan")
            for buf in (layer.D, layer.dc, layer.dW, layer.G):
                buf.fill_(float("nan"))
            layer.load_inputs(torch.from_numpy(X).to(BF).cuda())
            n0 = ard.ard_launch_count(ctx.h)
            h = layer.forward(1.5)
            n1 = ard.ard_launch_count(ctx.h)
            dX, dW = layer.backward(1.5, torch.from_numpy(dH).cuda())
            n2 = ard.ard_launch_count(ctx.h)
            tag = (dp, b)
            assert ard.ard_last_device_status(ctx.h) == 0, tag
            # one recurrence and one product, or one per gate
            assert n1 - n0 in (2, 5), tag
            assert (n2 - n1 in (3, 6, 9)) == bool(fits), (tag, n2 - n1)
            assert OG.rel_fro(host(h.float()), fw["Hs"]) <= TOL[ard.ARD_BF16], tag
            assert bool(torch.all(h[:, :, torch.from_numpy(m == 0).cuda()] == 0)), tag
            assert OG.rel_fro(host(dX), bw["dX"]) <= TOL[ard.ARD_BF16], tag
            assert OG.rel_fro(host(dW), bw["dW"].T) <= TOL[ard.ARD_BF16], tag
            kidx = torch.from_numpy(keep).cuda()
            assert OG.rel_fro(host(layer.D[0, :, I:][:, kidx]), bw["dh0"][:, keep]) <= TOL[ard.ARD_BF16], tag
            assert OG.rel_fro(host(layer.dc[:, :len(keep)]), bw["dc0"][:, keep]) <= TOL[ard.ARD_BF16], tag
    finally:
        ctx.close()
