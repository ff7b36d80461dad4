"""Recurrences inside clusters of CTAs, what the layer's own calls leave out: upstream gradients prepared in D and dc, states to begin from,
the caller's copy of the gate gradients (rows off the 16-byte grid), zeros of dropped rows beside columns of dW that stay, one to three
groups of 8 rows with a ragged last cluster; and the gate functions against 64 bits."""
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
ALPHA = 1.5


def _dev(a, dtype=F32):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(dtype).cuda()


def _gradients(fw, W, m, dH, dcT):
    """Gate gradients dZ [T][B][4H] and total gradients of h_{-1} .. h_{T-1} without h_{-1}'s mask."""
    T, B, H = dH.shape
    W = W.astype(np.float64)
    dZ, total = np.zeros((T, B, 4 * H)), np.zeros((T + 1, B, H))
    total[1:] = dH
    dc = dcT.astype(np.float64)
    for t in reversed(range(T)):
        _, i, f, g, o, c_prev, c = fw["saved"][t]
        dZ[t], dc = OL.cell_bwd(i, f, g, o, c_prev, c, m, ALPHA, total[t + 1], dc)
        total[t] += dZ[t] @ W[-H:].T
    return dZ, total


@pytest.mark.parametrize("T,B,I,H,dp,b", [
    (3, 127, 20, 380, 1, 1), (3, 60, 36, 508, 1, 1), (2, 127, 36, 508, 1, 1), (2, 61, 28, 764, 1, 1), (3, 113, 28, 764, 1, 1),
    (2, 37, 44, 1020, 2, 2), (10, 11, 20, 540, 3, 2), (3, 9, 24, 132, 3, 2), (2, 128, 64, 1024, 2, 1), (3, 5, 1064, 512, 16, 5)])
def test_prepared_gradients_and_the_recurrent_half(T, B, I, H, dp, b):
    KH, tol = I + H, TOL[ard.ARD_BF16]
    rng = np.random.default_rng(T * 1000 + B + H)
    m, keep = OP.row_mask(H, dp, b), OP.row_keep(H, dp, b)
    n, drop = len(keep), np.where(m == 0)[0]
    W = inputs.bf16_round(rng.uniform(-0.06, 0.06, size=(KH, 4 * H)).astype(np.float32))
    X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
    h0 = inputs.bf16_round((rng.uniform(-1, 1, size=(B, H)) * m[None, :]).astype(np.float32))
    c0 = (rng.uniform(-1, 1, size=(B, H)) * m[None, :]).astype(np.float32)
    dH = (rng.standard_normal((T, B, H)) / 8).astype(np.float32)
    dcT, d0 = ((rng.standard_normal((B, H)) / 8).astype(np.float32) for _ in range(2))
    fw = OL.fwd(X, W, None, m, ALPHA, h0=h0, c0=c0)
    bw = OL.bwd(fw, W, m, ALPHA, dH, dcT=dcT)
    dZ, total = _gradients(fw, W, m, dH, dcT)
    rows = torch.from_numpy(np.concatenate([g * H + drop for g in range(4)])).cuda()
    ctx = Ctx(1 << 20)
    try:
        pat = ctx.pattern(ard.ARD_ROW, KH, H)
        ard.ard_pattern_set(ctx.h, pat, dp, b)
        Wd, dh_last = _dev(W.T, BF), _dev(dH[T - 1])
        XH = torch.zeros((T + 1, B, KH), dtype=BF, device="cuda")
        XH[:T, :, :I], XH[0, :, I:] = _dev(X, BF), _dev(h0, BF)
        C = torch.zeros((T + 1, B, H), dtype=F32, device="cuda")
        C[0, :, :n] = _dev(c0[:, keep])
        G, Z = torch.zeros((T, B, 4 * H), dtype=F32, device="cuda"), torch.zeros((B, 4 * H), dtype=F32, device="cuda")
        ard.ard_lstm_forward(ctx.h, pat, T, B, I, H, ALPHA, XH, Wd, KH, None, C, G, Z)
        assert OG.rel_fro(host(XH[1:, :, I:].float()), fw["Hs"]) <= tol
        assert OG.rel_fro(host(C[T, :, :n]), fw["cT"][:, keep]) <= tol
        for recurrent in (0, 1):
            D, dc = torch.zeros((T, B, KH), dtype=F32, device="cuda"), torch.zeros((B, H), dtype=F32, device="cuda")
            D[1:, :, I:], D[0, :, I:], dc[:, :n] = _dev(dH[:-1]), _dev(d0), _dev(dcT[:, keep])
            DZ = torch.full((T, B, 4 * H), float("nan"), dtype=BF, device="cuda")
            dW = torch.full((4 * H, KH), float("nan"), dtype=F32, device="cuda")
            call = ard.ard_lstm_backward_recurrent if recurrent else ard.ard_lstm_backward
            call(ctx.h, pat, T, B, I, H, ALPHA, XH, Wd, KH, C, G, dh_last, D, dc, DZ, dW)
            assert ard.ard_last_device_status(ctx.h) == 0
            assert OG.rel_fro(host(dW[:, I:]), bw["dW"].T[:, I:]) <= tol, recurrent
            assert bool((dW[rows][:, I:] == 0).all()), recurrent
            if recurrent:
                assert bool(dW[:, :I].isnan().all())
                got = np.concatenate([host(DZ.float())[:, :, g * H:g * H + n] for g in range(4)], axis=2)
                want = np.concatenate([dZ[:, :, g * H + keep] for g in range(4)], axis=2)
                assert OG.rel_fro(got, want) <= tol
            else:
                assert OG.rel_fro(host(dW[:, :I]), bw["dW"].T[:, :I]) <= tol
                assert bool((dW[rows][:, :I] == 0).all())
                assert OG.rel_fro(host(D[:, :, :I]), bw["dX"]) <= tol
            got = host(D[:, :, I:])[:, :, keep]
            assert OG.rel_fro(got[0], (total[0] + d0)[:, keep]) <= tol, recurrent
            if T > 1:
                assert OG.rel_fro(got[1:], total[1:T][:, :, keep]) <= tol, recurrent
            assert OG.rel_fro(host(dc[:, :n]), bw["dc0"][:, keep]) <= tol, recurrent
    finally:
        ctx.close()


@pytest.mark.parametrize("refuse", [0, 1])  # in clusters, over the whole grid
def test_gate_functions(refuse):
    """One step from zero states with a zero weight: the gates are functions of the bias.  tanh within 2 ulps; the sigmoid 1 / (1 + e) with
    e = __expf(-x), whose documented error is 2 + 1.173 |x| ulps of 2^-23, and two more for the sum and the quotient.  (0 / 0 and the like
    would show as NaN.)"""
    T, B, I, H = 1, 3, 8, 768
    x = np.concatenate([np.logspace(-30, 2, 300), np.linspace(0.15, 0.19, 41), np.linspace(0.3, 12, 30),
                        [9.0, 9.1, 10.0, 10.5, 87.0, 88.5, 89.0, 104.0]]).astype(np.float32)
    x = np.concatenate([x, -x, np.float32([0.0, -0.0, np.inf, -np.inf, np.nan])])
    x = np.concatenate([x, np.linspace(-1, 1, H - len(x)).astype(np.float32)])
    ctx = Ctx(1 << 20)
    try:
        ard.ard_set_option(ctx.h, ard.ARD_OPT_LSTM_REFUSE, refuse)
        pat = ctx.pattern(ard.ARD_ROW, I + H, H)
        W, XH = torch.zeros((4 * H, I + H), dtype=BF, device="cuda"), torch.zeros((T + 1, B, I + H), dtype=BF, device="cuda")
        C = torch.zeros((T + 1, B, H), dtype=F32, device="cuda")
        G, Z = torch.zeros((T, B, 4 * H), dtype=F32, device="cuda"), torch.zeros((B, 4 * H), dtype=F32, device="cuda")
        ard.ard_lstm_forward(ctx.h, pat, T, B, I, H, 1.0, XH, W, I + H, _dev(np.tile(x, 4)), C, G, Z)
        assert ard.ard_last_device_status(ctx.h) == 0
        got = host(G).reshape(B, 4, H)
    finally:
        ctx.close()
    x64 = x.astype(np.float64) + 0.0  # the pre-activation is a sum: of -0 and the product's +0 it is +0
    with np.errstate(over="ignore", invalid="ignore"):
        tanh, sig = np.tanh(x64), 1.0 / (1.0 + np.exp(-x64))
        ok = np.isfinite(x64)
        spacing = np.spacing(np.abs(tanh).astype(np.float32)).astype(np.float64)
        for r in range(B):
            assert np.all(np.isnan(got[r][:, np.isnan(x64)]))
            g = got[r, 2]
            assert np.all(np.abs(g - tanh)[ok] <= 2 * spacing[ok]) and np.all(g[np.isinf(x64)] == np.sign(x64[np.isinf(x64)]))
            assert np.all(np.signbit(g[~np.isnan(x64)]) == np.signbit(x64[~np.isnan(x64)]))
            for gate in (0, 1, 3):
                s = got[r, gate]
                assert np.all(np.abs(s - sig)[ok] <= (4 + 1.25 * np.abs(x64[ok])) * 2.0 ** -23 * sig[ok] + 2.0 ** -126)
                assert np.all(s[np.isinf(x64)] == sig[np.isinf(x64)])
