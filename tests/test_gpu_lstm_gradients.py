"""What a backward pass leaves beside dX and dW, from buffers that held something else: the gradient of h_0 with zeros at its
dropped units, the gradient of c_0 with zeros behind the kept columns.  The step-by-step form of the same pass is the
reference."""
import numpy as np
import pytest
import torch

from oracle import pattern as OP
from paper_2203_05705_b200 import ard, inputs
from paper_2203_05705_b200.lstm import LstmLayer
from gpu_helpers import Ctx, TOL

pytestmark = pytest.mark.gpu
BF = torch.bfloat16


# shared and whole contractions of the gradients, on and off the 16-byte grid, one step, 12 units per CTA
@pytest.mark.parametrize("T,B,I,H", [(4, 20, 64, 128), (3, 33, 57, 131), (1, 9, 24, 40), (3, 70, 64, 1024), (2, 20, 36, 1300)])
def test_buffers_after_a_backward_pass(T, B, I, H):
    rng = np.random.default_rng(T + B + H)
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(4 * H, I + H)).astype(np.float32))
    X = torch.from_numpy(rng.standard_normal((T, B, I)).astype(np.float32)).to(BF).cuda()
    dH = torch.from_numpy((rng.standard_normal((T, B, H)) / 8).astype(np.float32)).cuda()
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, T, B, I, H, torch.from_numpy(W).to(BF).cuda())
        for dp, b in [(1, 1), (2, 2), (3, 1), (9, 5)]:
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            keep = torch.from_numpy(OP.row_keep(H, dp, b)).cuda()
            drop = torch.ones(H, dtype=torch.bool, device="cuda")
            drop[keep] = False
            res = []
            for persistent in (0, 1):
                ard.ard_set_lstm_persistent(ctx.h, persistent)
                layer.load_inputs(X)
                layer.forward(1.5)
                layer.D.fill_(float("nan"))
                layer.dc.fill_(float("nan"))
                layer.backward(1.5, dH)
                assert ard.ard_last_device_status(ctx.h) == 0
                res.append((layer.D[0, :, I:].double(), layer.dc.double()))
            (D0, c0), (D1, c1) = res
            n = len(keep)
            assert (D1[:, keep] - D0[:, keep]).norm() <= TOL[ard.ARD_BF16] * D0[:, keep].norm(), dp
            assert (c1[:, :n] - c0[:, :n]).norm() <= TOL[ard.ARD_BF16] * c0[:, :n].norm(), dp
            assert bool((c0[:, n:] == 0).all()) and bool((c1[:, n:] == 0).all()), dp
            assert bool((D1[:, drop] == 0).all()), dp
    finally:
        ctx.close()


# 148 SMs hold 38.8 MB of gate gradients in context scratch (T * B * 4 * H bf16, H rounded up to 8) for layers whose own are off
# the 16-byte grid: the last length that fits and the first that does not; and a layer off the grid for its inputs alone, whose
# gate gradients need no copy however many there are
@pytest.mark.parametrize("T,I,H,one_kernel", [(34, 20, 1092, True), (35, 20, 1092, False), (35, 20, 1096, True)])
def test_gate_gradients_around_the_limit_of_the_scratch(T, I, H, one_kernel):
    B = 128
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the scratch is sized by the number of SMs")
    g = torch.Generator(device="cuda").manual_seed(T + H)
    W = (torch.rand((4 * H, I + H), device="cuda", generator=g) * 0.12 - 0.06).to(BF)
    X = torch.randn((T, B, I), device="cuda", generator=g).to(BF)
    dH = torch.randn((T, B, H), device="cuda", generator=g) / 8
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        layer = LstmLayer(ctx.h, pat, T, B, I, H, W)
        ard.ard_pattern_set(ctx.h, pat, 2, 2)
        res = []
        for persistent in (0, 1):
            ard.ard_set_lstm_persistent(ctx.h, persistent)
            layer.load_inputs(X)
            layer.forward(1.5)
            n0 = ard.ard_launch_count(ctx.h)
            dX, dW = layer.backward(1.5, dH)
            n = ard.ard_launch_count(ctx.h) - n0
            assert (n <= 9) == (bool(persistent) and one_kernel), n
            assert ard.ard_last_device_status(ctx.h) == 0
            res.append((dX.double().clone(), dW.double().clone()))
        for a, r in zip(res[1], res[0]):
            assert (a - r).norm() <= TOL[ard.ARD_BF16] * r.norm()
    finally:
        ctx.close()
