"""Whole-sequence LSTM calls whose launches the device refuses, for patterns on both sides of what the clusters hold while the host knows
neither: a refused call has enqueued nothing before it takes another way, so operands that are input and output at once (the upstream
gradients in D, dc, the pre-activations in G) enter once."""
import numpy as np
import pytest
import torch

from oracle import gemm as OG
from oracle import lstm as OL
from oracle import pattern as OP
from paper_2203_05705_b200 import ard, inputs
from gpu_helpers import Ctx, host, TOL

pytestmark = pytest.mark.gpu
BF, F32 = torch.bfloat16, torch.float32
T, B, I, H = 3, 9, 40, 1024
KH = I + H
ALPHA = 1.5


def _dev(a, dtype=F32):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(dtype).cuda()


class Layer:
    """A layer after its forward pass, with operands of the backward calls that nothing in them is zero of."""

    def __init__(self, ctx, dp):
        K = [0.5, 0.5]
        ard.ard_set_distribution(ctx.h, 0, K)
        cdf = OP.quantise_K(K)
        it = next(i for i in range(1000) if OP.draw(cdf, 5, i, 0)[0] == dp)
        self.pat = ctx.pattern(ard.ARD_ROW, KH, H)
        ard.ard_sample_pattern(ctx.h, self.pat, 0, 5, it, 0)
        rng = np.random.default_rng(dp)
        b = OP.draw(cdf, 5, it, 0)[1]
        m, self.keep = OP.row_mask(H, dp, b), OP.row_keep(H, dp, b)
        self.n = len(self.keep)
        W = inputs.bf16_round(rng.uniform(-0.05, 0.05, size=(KH, 4 * H)).astype(np.float32))
        X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
        h0 = inputs.bf16_round((rng.uniform(-1, 1, size=(B, H)) * m[None, :]).astype(np.float32))
        c0 = (rng.uniform(-1, 1, size=(B, H)) * m[None, :]).astype(np.float32)
        dH = (rng.standard_normal((T, B, H)) / 8).astype(np.float32)
        dcT = (rng.standard_normal((B, H)) / 8).astype(np.float32)
        d0 = (rng.standard_normal((B, H)) / 8).astype(np.float32)
        self.fw = OL.fwd(X, W, None, m, ALPHA, h0=h0, c0=c0)
        self.bw = OL.bwd(self.fw, W, m, ALPHA, dH, dcT=dcT)
        self.want_d0 = self.bw["dh0"] + d0
        self.W = _dev(W.T, BF)
        self.XH = torch.zeros((T + 1, B, KH), dtype=BF, device="cuda")
        self.XH[:T, :, :I] = _dev(X, BF)
        self.XH[0, :, I:] = _dev(h0, BF)
        self.C = torch.zeros((T + 1, B, H), dtype=F32, device="cuda")
        self.C[0, :, :self.n] = _dev(c0[:, self.keep])
        self.G = torch.zeros((T, B, 4 * H), dtype=F32, device="cuda")
        self.Z = torch.zeros((B, 4 * H), dtype=F32, device="cuda")
        self.D = torch.zeros((T, B, KH), dtype=F32, device="cuda")
        self.D[1:, :, I:] = _dev(dH[:-1])
        self.D[0, :, I:] = _dev(d0)
        self.dh_last = _dev(dH[T - 1])
        self.dc = torch.zeros((B, H), dtype=F32, device="cuda")
        self.dc[:, :self.n] = _dev(dcT[:, self.keep])
        self.DZ = torch.zeros((T, B, 4 * H), dtype=BF, device="cuda")
        self.dW = torch.full((4 * H, KH), float("nan"), dtype=F32, device="cuda")

    def forward(self, ctx):
        ard.ard_lstm_forward(ctx.h, self.pat, T, B, I, H, ALPHA, self.XH, self.W, KH, None, self.C, self.G, self.Z)

    def backward_args(self, ctx):
        return (ctx.h, self.pat, T, B, I, H, ALPHA, self.XH, self.W, KH, self.C, self.G, self.dh_last, self.D, self.dc, self.DZ, self.dW)


@pytest.mark.parametrize("dp", [1, 2])
@pytest.mark.parametrize("refuse", [0, 1, 2, 3])
def test_prepared_gradients_enter_once(refuse, dp):
    ctx = Ctx(1 << 20)
    try:
        y = Layer(ctx, dp)
        tol = TOL[ard.ARD_BF16]
        ard.ard_set_option(ctx.h, ard.ARD_OPT_LSTM_REFUSE, refuse)
        y.forward(ctx)
        assert OG.rel_fro(host(y.XH[1:, :, I:].float()), y.fw["Hs"]) <= tol
        assert OG.rel_fro(host(y.C[T, :, :y.n]), y.fw["cT"][:, y.keep]) <= tol
        ard.ard_lstm_backward(*y.backward_args(ctx))
        assert ard.ard_last_device_status(ctx.h) == 0
        assert OG.rel_fro(host(y.D[:, :, :I]), y.bw["dX"]) <= tol
        assert OG.rel_fro(host(y.dW), y.bw["dW"].T) <= tol
        assert OG.rel_fro(host(y.D[0, :, I:])[:, y.keep], y.want_d0[:, y.keep]) <= tol
        assert OG.rel_fro(host(y.dc[:, :y.n]), y.bw["dc0"][:, y.keep]) <= tol
    finally:
        ctx.close()


@pytest.mark.parametrize("dp", [1, 2])
@pytest.mark.parametrize("refuse", [2, 3])
def test_calls_without_another_way_leave_their_operands_alone(refuse, dp):
    ctx = Ctx(1 << 20)
    try:
        y = Layer(ctx, dp)
        y.forward(ctx)
        held = [t.clone() for t in (y.XH, y.C, y.G, y.D, y.dc, y.DZ)]
        ard.ard_set_option(ctx.h, ard.ARD_OPT_LSTM_REFUSE, refuse)
        with pytest.raises(ard.ArdError):
            ard.ard_lstm_backward_recurrent(*y.backward_args(ctx))
        with pytest.raises(ard.ArdError):
            ard.ard_lstm_forward_from_gates(ctx.h, y.pat, T, B, I, H, ALPHA, y.XH, y.W, KH, None, y.C, y.G)
        assert ard.ard_last_device_status(ctx.h) == 0
        for t, was in zip((y.XH, y.C, y.G, y.D, y.dc, y.DZ), held):
            assert torch.equal(t, was)
        assert bool(y.dW.isnan().all())
    finally:
        ctx.close()


@pytest.mark.parametrize("compact,launches", [(0, 2), (1, 3)])
def test_kernels_that_the_option_rules_out_are_not_enqueued(compact, launches):
    ctx = Ctx(1 << 20)
    try:
        y = Layer(ctx, 2)
        ard.ard_set_option(ctx.h, ard.ARD_OPT_LSTM_COMPACT_H, compact)
        n0 = ard.ard_launch_count(ctx.h)
        y.forward(ctx)
        n1 = ard.ard_launch_count(ctx.h)
        ard.ard_lstm_backward(*y.backward_args(ctx))
        # the product of the input half and one recurrence or two; and the weight gradient
        assert (n1 - n0, ard.ard_launch_count(ctx.h) - n1) == (launches, launches + 1)
        assert OG.rel_fro(host(y.XH[1:, :, I:].float()), y.fw["Hs"]) <= TOL[ard.ARD_BF16]
        assert OG.rel_fro(host(y.dW), y.bw["dW"].T) <= TOL[ard.ARD_BF16]
        assert ard.ard_last_device_status(ctx.h) == 0
    finally:
        ctx.close()


def test_the_option_takes_two_bits():
    ctx = Ctx(1 << 20)
    try:
        for bad in (-1, 4):
            with pytest.raises(ard.ArdError):
                ard.ard_set_option(ctx.h, ard.ARD_OPT_LSTM_REFUSE, bad)
    finally:
        ctx.close()
