"""A pattern that a captured call draws: replays draw it again where the host does not see it, so what an ordinary call set last says
nothing about what a later LSTM call finds."""
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


@pytest.mark.parametrize("persistent", [1, 0])
def test_a_pattern_drawn_by_a_captured_iteration_of_a_stack(persistent):
    T, B, I, H, out = 2, 8, 40, 512, 8
    KH, alpha = I + H, 1.5
    rng = np.random.default_rng(11)
    K = [0.5] + [0.0] * 6 + [0.5]
    cdf = OP.quantise_K(K)
    zeros = lambda *shape, dtype=BF: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    W = inputs.bf16_round(rng.uniform(-0.08, 0.08, size=(KH, 4 * H)).astype(np.float32))
    X = inputs.bf16_round(rng.standard_normal((T, B, I)).astype(np.float32))
    Wd = torch.from_numpy(np.ascontiguousarray(W.T)).to(BF).cuda()
    ctx = Ctx(1 << 20)
    try:
        ard.ard_set_option(ctx.h, ard.ARD_OPT_MLP_PERSISTENT, persistent)
        ard.ard_set_distribution(ctx.h, 0, K)
        layers = []
        for k, n, hidden in ((KH, H, 1), (H, out, 0)):
            layers.append(dict(K=k, N=n, pat=ctx.pattern(ard.ARD_ROW, k, n), sample=hidden, relu=hidden, compact_out=hidden, dW_is_f32=0,
                               alpha=1.0, ldw=k, W=torch.randn((n, k), device="cuda").to(BF), bias=None, Wk=zeros(n, k), A=zeros(B, n),
                               dZ=zeros(B, n), dWk=zeros(n, k), dW=zeros(n, k), db=zeros(n, dtype=F32)))
        pat = layers[0]["pat"]
        table = ard.mlp_layers(layers)
        x, d_out, dx = zeros(B, KH), zeros(B, out), zeros(B, KH)
        counter = torch.zeros(1, dtype=torch.int64, device="cuda")
        s = torch.cuda.Stream()
        torch.cuda.synchronize()

        def step():
            ard.ard_mlp_step(ctx.h, table, 2, B, x, KH, d_out, out, dx, KH, 0, 21, 0, counter, s.cuda_stream)

        step()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            step()
        ard.ard_pattern_set(ctx.h, pat, 8, 1, s.cuda_stream)
        it = 1
        with torch.cuda.stream(s):
            while True:  # a replay that draws a period of 1
                g.replay()
                dp, b = OP.draw(cdf, 21, it, 1)
                it += 1
                if dp == 1:
                    break
        torch.cuda.synchronize()
        got = ard.ard_pattern_to_host(pat, H)
        assert (got[0], got[1], got[2]) == (1, 1, H)
        XH = zeros(T + 1, B, KH)
        XH[:T, :, :I] = torch.from_numpy(X).to(BF).cuda()
        C, G, Z = zeros(T + 1, B, H, dtype=F32), zeros(T, B, 4 * H, dtype=F32), zeros(B, 4 * H, dtype=F32)
        ard.ard_lstm_forward(ctx.h, pat, T, B, I, H, alpha, XH, Wd, KH, None, C, G, Z)
        assert ard.ard_last_device_status(ctx.h) == 0
        fw = OL.fwd(X, W, None, OP.row_mask(H, 1, 1), alpha)
        assert OG.rel_fro(host(XH[1:, :, I:].float()), fw["Hs"]) <= TOL[ard.ARD_BF16]
        del g
    finally:
        ctx.close()
