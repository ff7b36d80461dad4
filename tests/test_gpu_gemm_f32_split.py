"""fp32 layers large enough for the tensor cores (operands split into three bf16 parts) against the oracle: edges of the 128 x 64
tiles and of the contraction blocks, rows on and off the 16-byte grid, cut and whole contractions, a compact copy of dY or none,
operands and sums that are not finite, very small or of one sign."""
import numpy as np
import pytest
import torch

from paper_2203_05705_b200 import ard
from gpu_helpers import Ctx, run_three_gemms, assert_ok, oracle_mask

pytestmark = pytest.mark.gpu

# What is left out of a product of two elements is below 2^-25 of it; sums of 64 products lose up to four truncations (2^-22 of a
# partial sum) and are added with round to nearest.  The operands are random, so the errors of a sum's terms are too: 1e-6.
TOL = 1e-6


def _layer(B, K, N):
    rng = np.random.default_rng(B + K + N)
    X, W, dY = (rng.standard_normal(s).astype(np.float32) for s in ((B, K), (K, N), (B, N)))
    return X, W / np.float32(np.sqrt(K)), dY


# contractions cut eight, four and two ways and not at all
ROWS = [(250, 4099, 510), (250, 510, 4099), (4099, 250, 510), (257, 2051, 701), (385, 3001, 1003), (513, 2087, 1531)]
TILES = [(32, 700, 36, 35), (12, 800, 90, 101), (128, 520, 9, 10), (200, 520, 6, 7), (4, 500, 300, 300)]


@pytest.mark.parametrize("B,K,N", [(128, 2048, 2048), (129, 2087, 1531), (5, 6001, 8193), (4097, 65, 1201), (4100, 700, 130)] + ROWS)
@pytest.mark.parametrize("workspace", [0, 32 << 20])
def test_row_pattern(B, K, N, workspace):
    X, W, dY = _layer(B, K, N)
    ctx = Ctx(workspace)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        for i, (dp, b) in enumerate([(1, 1), (2, 2), (3, 1)]):
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_F32, X, W, dY, dp, b, 1.5, compact=(i == 1), zero_fill=(i != 2),
                                  lds={"x": K + i, "w": (K + 3) // 4 * 4, "y": N + 5 * (i & 1)})
            assert_ok(res, TOL, (B, K, N, dp, b))
    finally:
        ctx.close()


@pytest.mark.parametrize("ts,B,Tr,Tc", [(32, 129, 64, 33), (12, 200, 90, 101), (128, 260, 9, 10), (200, 130, 6, 7)] + TILES)
def test_tile_pattern(ts, B, Tr, Tc):
    K, N = Tr * ts, Tc * ts
    X, W, dY = _layer(B, K, N)
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_TILE, K, N, ts)
        for i, dp in enumerate([1, 2, 3, 5]):
            b = 1 + i % dp
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            res = run_three_gemms(ctx, pat, ard.ARD_TILE, ard.ARD_F32, X, W, dY, dp, b, 2.0, ts=ts, zero_fill=(i % 2 == 0),
                                  lds={"x": K + 4 * (i & 1), "w": K, "y": N + i // 3})
            assert_ok(res, TOL, (ts, B, Tr, Tc, dp, b))
    finally:
        ctx.close()


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.395e38])
@pytest.mark.parametrize("kind,ts,dp", [(ard.ARD_ROW, 0, 1), (ard.ARD_ROW, 0, 2), (ard.ARD_TILE, 64, 3)])
@pytest.mark.parametrize("B", [200, 700])
def test_not_finite(value, kind, ts, dp, B):
    """An infinity, a NaN or a value that no bf16 holds ends up where the CUDA-core kernel has it."""
    K, N = 1536, 1088
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(kind, K, N, ts)
        ard.ard_pattern_set(ctx.h, pat, dp, 1)
        for where in range(3):
            g = torch.Generator(device="cuda").manual_seed(where)
            ops = [torch.randn(s, device="cuda", generator=g) * 0.1 for s in ((B, K), (N, K), (B, N))]
            ops[where][130, 66 if where == 2 else 700] = value  # row 130 of the weight and column 66 of dY are kept neurons
            X, W, dY = ops
            outs = []
            for path in (ard.ARD_PATH_CUDA_CORE, ard.ARD_PATH_AUTO):
                ard.ard_set_path(ctx.h, path)
                Y, dX, dW = (torch.full(s, 7.0, device="cuda") for s in ((B, N), (B, K), (N, K)))
                ard.ard_fwd(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, X, K, W, K, Y, N, ard.ARD_OUT_SCATTER_ZEROFILL)
                ard.ard_bwd_data(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, dY, N, 0, W, K, dX, K)
                ard.ard_bwd_weight(ctx.h, pat, ard.ARD_F32, ard.ARD_F32, B, K, N, 1.0, X, K, dY, N, 0, dW, K, 1)
                outs.append([Y, dX, dW])
            for cc, tc in zip(*outs):
                fin = cc.isfinite()
                assert torch.equal(fin, tc.isfinite()) and torch.equal(cc.isnan(), tc.isnan()) and torch.equal(cc[cc.isinf()], tc[tc.isinf()])
                assert (cc[fin].double() - tc[fin].double()).norm() <= 2e-6 * cc[fin].double().norm()
    finally:
        ctx.close()


def _both_paths(ctx, pat, B, K, N, X, W, dY, relu=False):
    outs = []
    for path in (ard.ARD_PATH_CUDA_CORE, ard.ARD_PATH_AUTO):
        ard.ard_set_path(ctx.h, path)
        Y, dX, dW = (torch.full(s, 7.0, device="cuda") for s in ((B, N), (B, K), (N, K)))
        if relu:
            ard.ard_layer_fwd(ctx.h, pat, None, ard.ARD_F32, B, K, N, 1.0, X, K, W, K, None, Y, N,
                              ard.ARD_OUT_SCATTER_ZEROFILL | ard.ARD_FLAG_RELU)
        else:
            ard.ard_fwd(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, X, K, W, K, Y, N, ard.ARD_OUT_SCATTER_ZEROFILL)
        ard.ard_bwd_data(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, dY, N, 0, W, K, dX, K)
        ard.ard_bwd_weight(ctx.h, pat, ard.ARD_F32, ard.ARD_F32, B, K, N, 1.0, X, K, dY, N, 0, dW, K, 1)
        outs.append([Y, dX, dW])
    return list(zip(*outs))


@pytest.mark.parametrize("x,w", [(1e30, 1e30), (-1e25, 3e20), (3e20, -1e25), (2.0 ** 64 * (1 - 2 ** -10), 2.0 ** 64 * (1 - 2 ** -10)),
                                 (2.0 ** 70 * (1 - 2 ** -10), 2.0 ** 70 * (1 - 2 ** -10)), (2.0 ** 63 * (2 - 2 ** -9), 2.0 ** 64 * (1 - 2 ** -20))])
@pytest.mark.parametrize("kind,ts,dp,relu", [(ard.ARD_ROW, 0, 1, False), (ard.ARD_ROW, 0, 2, True), (ard.ARD_TILE, 64, 3, False)])
def test_products_near_and_beyond_the_largest_number(x, w, kind, ts, dp, relu):
    """Finite operands whose product overflows, or only just does not: as the CUDA-core kernel has it."""
    B, K, N = 700, 1536, 1088
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(kind, K, N, ts)
        ard.ard_pattern_set(ctx.h, pat, dp, 1)
        g = torch.Generator(device="cuda").manual_seed(1)
        X, W, dY = (torch.randn(s, device="cuda", generator=g) * 0.1 for s in ((B, K), (N, K), (B, N)))
        X[130, 700], dY[130, 66], W[66, 700] = x, x, w  # kept under every pattern here
        for cc, tc in _both_paths(ctx, pat, B, K, N, X, W, dY, relu):
            fin = cc.isfinite()
            assert not tc.isnan().any() and torch.equal(fin, tc.isfinite()) and torch.equal(cc[~fin], tc[~fin])
            assert (cc[fin].double() - tc[fin].double()).norm() <= 2e-6 * cc[fin].double().norm()
        assert ard.ard_last_device_status(ctx.h) == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("B,K,N,kind,ts,dp", [(513, 2087, 1531, ard.ARD_ROW, 0, 1), (513, 2087, 1531, ard.ARD_ROW, 0, 2),
                                              (4099, 250, 510, ard.ARD_ROW, 0, 1), (800, 1080, 1212, ard.ARD_TILE, 12, 1),
                                              (500, 1200, 1200, ard.ARD_TILE, 4, 5)])
def test_not_finite_at_the_edges(B, K, N, kind, ts, dp):
    """Infinities in the last row, column and index of ragged tiles: what the repeated products read and write."""
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(kind, K, N, ts)
        ard.ard_pattern_set(ctx.h, pat, dp, 1)
        X, W, dY = (torch.randn(s, device="cuda") * 0.1 for s in ((B, K), (N, K), (B, N)))
        last = (N - 1) // dp * dp if kind == ard.ARD_ROW else N - 1  # kept neuron
        X[-1, -1] = X[0, 0] = float("inf")
        W[last, -1], dY[-1, last], dY[0, 0] = float("-inf"), float("inf"), float("nan")
        for cc, tc in _both_paths(ctx, pat, B, K, N, X, W, dY):
            fin = cc.isfinite()
            assert torch.equal(fin, tc.isfinite()) and torch.equal(cc.isnan(), tc.isnan()) and torch.equal(cc[cc.isinf()], tc[tc.isinf()])
            assert (cc[fin].double() - tc[fin].double()).norm() <= 2e-6 * cc[fin].double().norm()
        assert ard.ard_last_device_status(ctx.h) == 0
    finally:
        ctx.close()


def test_not_finite_in_a_long_contraction():
    """A weight gradient over a million rows, its contraction not cut: the repeat ends well before the kernel's waits give up."""
    B, K, N = 1 << 20, 1216, 512
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        ard.ard_pattern_set(ctx.h, pat, 1, 1)
        X, dY = torch.full((B, K), 0.5, device="cuda"), torch.full((B, N), 0.25, device="cuda")
        X[B // 2, 1] = dY[7, 2] = float("nan")
        dW = torch.zeros((N, K), device="cuda")
        ard.ard_bwd_weight(ctx.h, pat, ard.ARD_F32, ard.ARD_F32, B, K, N, 1.0, X, K, dY, N, 0, dW, K, 1)
        assert ard.ard_last_device_status(ctx.h) == 0
        want = torch.full((N, K), 0.125 * B, device="cuda")  # exact in fp32
        want[:, 1] = want[2, :] = float("nan")
        assert torch.equal(want.isnan(), dW.isnan()) and torch.equal(want.nan_to_num(), dW.nan_to_num())
    finally:
        ctx.close()


@pytest.mark.parametrize("exponent", [-100, -113, -126, -140])
@pytest.mark.parametrize("kind,ts,dp", [(ard.ARD_ROW, 0, 1), (ard.ARD_TILE, 64, 3)])
def test_small_elements_keep_their_bits(exponent, kind, ts, dp):
    """Operands down to fp32's subnormal numbers (the others large enough for results that are not)."""
    B, K, N = 700, 1536, 1088
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(kind, K, N, ts)
        ard.ard_pattern_set(ctx.h, pat, dp, 1)
        mask = torch.from_numpy(np.ascontiguousarray(oracle_mask(kind, K, N, ts, dp, 1).T)).cuda().double()
        for where in range(3):
            ops = [torch.randn(s, device="cuda") * 2.0 ** (exponent if i == where else 30) for i, s in enumerate(((B, K), (N, K), (B, N)))]
            X, W, dY = [o.double() for o in ops]
            Wm = W * (mask if mask.ndim == 2 else mask[:, None])
            want = [X @ Wm.T, dY @ Wm, (dY.T @ X) * (mask if mask.ndim == 2 else mask[:, None])]
            for w, (_, tc) in zip(want, _both_paths(ctx, pat, B, K, N, *ops)):
                assert (tc.double() - w).norm() <= TOL * w.norm()
    finally:
        ctx.close()


@pytest.mark.parametrize("M,K,N", [(256, 4096, 512), (256, 512, 4096), (4096, 256, 512), (1024, 1024, 1024)])
def test_operands_of_one_sign(M, K, N):
    """Truncated sums of terms of one sign lose in one direction: still no larger an error than the CUDA-core kernel's (shapes whose
    contraction that one cuts eight ways among them, where its error is smallest)."""
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        ard.ard_pattern_set(ctx.h, pat, 1, 1)
        g = torch.Generator(device="cuda").manual_seed(K)
        for draw in (lambda s: torch.rand(s, device="cuda", generator=g), lambda s: torch.randn(s, device="cuda", generator=g).abs()):
            X, W, dY = draw((M, K)), draw((N, K)), draw((M, N))
            want = [X.double() @ W.double().T, dY.double() @ W.double(), dY.double().T @ X.double()]
            for w, (cc, tc) in zip(want, _both_paths(ctx, pat, M, K, N, X, W, dY)):
                assert (tc.double() - w).norm() <= (cc.double() - w).norm()
    finally:
        ctx.close()


def _tensors(B, K, N, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(s, device="cuda", generator=g) * (K ** -0.5 if i == 1 else 1.0) for i, s in enumerate(((B, K), (N, K), (B, N)))]


def test_the_compact_copy_is_not_kept_between_calls():
    """ard_set_compact_reuse is for bf16 calls: an fp32 layer's dY may be written between its two backward calls."""
    B, K, N = 1017, 2049, 1481
    ctx = Ctx(4 * B * (N + 8))
    try:
        ard.ard_set_compact_reuse(ctx.h, True)
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        ard.ard_pattern_set(ctx.h, pat, 2, 1)
        X, W, dY = _tensors(B, K, N)
        dX, dW = torch.zeros((B, K), device="cuda"), torch.zeros((N, K), device="cuda")
        ard.ard_bwd_data(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, dY, N, 0, W, K, dX, K)
        dY.mul_(-3.0)
        ard.ard_bwd_weight(ctx.h, pat, ard.ARD_F32, ard.ARD_F32, B, K, N, 1.0, X, K, dY, N, 0, dW, K, 1)
        want = dY.double().T @ X.double()
        want[1::2] = 0.0
        assert (dW.double() - want).norm() <= TOL * want.norm()
    finally:
        ctx.close()


@pytest.mark.parametrize("B,K,N,ts", [r + (0,) for r in ROWS] + [(B, Tr * ts, Tc * ts, ts) for ts, B, Tr, Tc in TILES])
def test_these_layers_reach_the_kernel(B, K, N, ts):
    """Other sums than the CUDA-core kernel's, bit for bit, from at least two of the three products."""
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_TILE if ts else ard.ARD_ROW, K, N, ts)
        ard.ard_pattern_set(ctx.h, pat, 1, 1)
        assert sum(not torch.equal(cc, tc) for cc, tc in _both_paths(ctx, pat, B, K, N, *_tensors(B, K, N))) >= 2
    finally:
        ctx.close()


# from 2e9 kept operations on the backward products of a row pattern read a compact copy of dY, where the workspace has room for it
COMPACTED = [(1017, 2049, 1481), (1030, 2052, 2308)]


@pytest.mark.parametrize("B,K,N", COMPACTED)
@pytest.mark.parametrize("room", [0, -1])
def test_compact_copy_of_a_full_width_gradient(B, K, N, room):
    X, W, dY = _layer(B, K, N)
    ctx = Ctx(4 * B * ((N + 7) // 8 * 8) + room)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        for dp, b in [(2, 2), (3, 1)]:
            ard.ard_pattern_set(ctx.h, pat, dp, b)
            before = ard.ard_launch_count(ctx.h)
            res = run_three_gemms(ctx, pat, ard.ARD_ROW, ard.ARD_F32, X, W, dY, dp, b, 1.5, lds={"y": N + 3})
            assert_ok(res, TOL, (B, K, N, dp, b))
            assert ard.ard_launch_count(ctx.h) - before in ((4, 5) if room == 0 else (3,))
    finally:
        ctx.close()


@pytest.mark.parametrize("side_streams", [0, 1])
def test_compact_copy_over_a_distribution(side_streams):
    """Dense draws of a distribution that drops something go through the copy too; ard_layer_products makes one for both products."""
    B, K, N = COMPACTED[1]
    ctx = Ctx(4 * B * (N + 8))
    try:
        ard.ard_set_option(ctx.h, ard.ARD_OPT_SIDE_STREAMS, side_streams)
        ard.ard_set_distribution(ctx.h, 0, [0.4, 0.3, 0.3])
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        X, W, dY = _tensors(B, K, N)
        seen = set()
        for it in range(12):
            ard.ard_sample_pattern(ctx.h, pat, 0, 1, it, 0)
            dp, _, _, keep = ard.ard_pattern_to_host(pat, N)
            if dp in seen:
                continue
            seen.add(dp)
            mask = torch.zeros(N, dtype=torch.float64, device="cuda")
            mask[torch.from_numpy(keep).long().cuda()] = 1.0
            dY.mul_(-1.5)  # another gradient in the same buffer
            Y, dX, dW = (torch.full(s, float("nan"), device="cuda") for s in ((B, N), (B, K), (N, K)))
            ard.ard_layer_products(ctx.h, pat, ard.ARD_F32, ard.ARD_F32, B, K, N, 2.0, X, K, W, K, dY, N, Y, N,
                                   ard.ARD_OUT_SCATTER_ZEROFILL, dX, K, dW, K, 1)
            dYm = dY.double() * mask
            for got, want in zip((Y, dX, dW), (X.double() @ W.double().T * mask, dYm @ W.double(), dYm.T @ X.double())):
                assert (got.double() - 2.0 * want).norm() <= TOL * 2.0 * want.norm(), dp
        assert seen == {1, 2, 3}
        assert ard.ard_last_device_status(ctx.h) == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("B,K,N", [(513, 2087, 1531), (700, 1536, 1088)])
def test_accumulate(B, K, N):
    """ARD_FLAG_ACCUMULATE: compact forward and input gradient added to what is there."""
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        X, W, dY = _tensors(B, K, N)
        for dp in (1, 2):
            ard.ard_pattern_set(ctx.h, pat, dp, 1)
            n = (N - 1) // dp + 1
            Y, dX = torch.randn((B, N), device="cuda"), torch.randn((B, K), device="cuda")
            wantY, wantdX = Y.double(), dX.double()
            wantY[:, :n] += X.double() @ W[::dp].double().T
            wantdX += dY[:, ::dp].double() @ W[::dp].double()
            ard.ard_fwd(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, X, K, W, K, Y, N, ard.ARD_OUT_COMPACT | ard.ARD_FLAG_ACCUMULATE)
            ard.ard_bwd_data(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, dY, N, ard.ARD_FLAG_ACCUMULATE, W, K, dX, K)
            for got, want in ((Y, wantY), (dX, wantdX)):
                assert (got.double() - want).norm() <= TOL * want.norm()
    finally:
        ctx.close()


def test_static_scratch():
    """The entry point without a workspace, at a size that the tensor cores take (B * N * 4 bytes fit its fixed array)."""
    B, K, N = 700, 2048, 1531
    ctx = Ctx(0)
    try:
        pat = ctx.pattern(ard.ARD_ROW, K, N)
        X, W, dY = _tensors(B, K, N)
        for dp in (1, 2):
            ard.ard_pattern_set(ctx.h, pat, dp, 1)
            outs = []
            for path in (ard.ARD_PATH_CUDA_CORE, ard.ARD_PATH_AUTO):
                ard.ard_set_path(ctx.h, path)
                dX = torch.full((B, K), float("nan"), device="cuda")
                ard.ard_bwd_data_static_scratch(ctx.h, pat, ard.ARD_F32, B, K, N, 1.0, dY, N, W, K, dX, K)
                outs.append(dX)
            want = dY[:, ::dp].double() @ W[::dp].double()
            assert (outs[1].double() - want).norm() <= TOL * want.norm()
            assert not torch.equal(*outs)  # not the CUDA-core kernel's sums
    finally:
        ctx.close()
