"""Performance cases of the framework: what its users have it do, at the sizes they do it.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)` one more of the same ranges,
`prepare(case, seed)` what a training program holds before the call (weights, inputs, buffers, the library's
context and pattern objects), `run(state)` one pass through the public entry points, `work(case)` the bytes and
operations such a pass cannot do without, `tolerance(case)` how far two correct implementations may differ.

Every pass is one training iteration: a pattern is drawn on the device with the counter-based sampler, a new one
in each pass.  The period `dp` is part of the case (the distribution handed to the library has its whole weight on
it), so that all passes of a case do the same amount of work; the offset is drawn.  A run over a distribution is the
mean over its periods: about a third of the iterations are dense (dp = 1) at a rate of one half, the rest spread
over 2 .. 16.

Kinds:
  layer        ard_fwd, ard_bwd_data, ard_bwd_weight of one layer ("calls": "three"), or ard_layer_products ("one")
  mlp          ard_mlp_step, a whole training iteration of a stack of layers
  lstm         lstm.LstmLayer: forward and backward over a sequence, dropout on the hidden units
  conv_rows    sensitivity prediction, row sampling and products over the kept rows of an im2col matrix
  conv_blocks  the same with blocks of the matrix as the granularity
"""
import math
import weakref

import torch

from paper_2203_05705_b200 import ard, lstm

SAMPLER_SEED = 20220305
N_PERIODS = 16  # longest period of the distributions
BF16, F32 = torch.bfloat16, torch.float32


def listed():
    return [
        # The tiny fp32 layer of the MNIST network's shape: the smallest calls, where launches and latency count.
        {"name": "fp32_784x256", "kind": "layer", "pattern": "row", "dtype": "f32", "calls": "three", "B": 64, "K": 784,
         "N": 256, "ts": 0, "dp": 2},
        # A hidden layer of the paper's MLP (batch 128, 2048 x 2048) kept in fp32, a dense iteration.
        {"name": "fp32_2048", "kind": "layer", "pattern": "row", "dtype": "f32", "calls": "three", "B": 128, "K": 2048,
         "N": 2048, "ts": 0, "dp": 1},
        # The same layer in bf16 under the paper's own 32 x 32 weight tiles.
        {"name": "tile32_2048", "kind": "layer", "pattern": "tile", "dtype": "bf16", "calls": "three", "B": 128,
         "K": 2048, "N": 2048, "ts": 32, "dp": 2},
        # Tile-based DropConnect of a 4096 x 4096 weight, batch 1024, 64 x 64 tiles.
        {"name": "tile64_4096", "kind": "layer", "pattern": "tile", "dtype": "bf16", "calls": "one", "B": 1024,
         "K": 4096, "N": 4096, "ts": 64, "dp": 4},
        # The large MLP layer, 8192 x 8192 at batch 4096: 128 x 128 tiles, and kept neurons.
        {"name": "tile128_8192", "kind": "layer", "pattern": "tile", "dtype": "bf16", "calls": "one", "B": 4096,
         "K": 8192, "N": 8192, "ts": 128, "dp": 3},
        {"name": "row_8192", "kind": "layer", "pattern": "row", "dtype": "bf16", "calls": "one", "B": 4096, "K": 8192,
         "N": 8192, "ts": 0, "dp": 2},
        # A layer between 1500-wide LSTM layers over the 20 x 35 positions of a batch: rows of 3000 bytes.
        {"name": "row_1500", "kind": "layer", "pattern": "row", "dtype": "bf16", "calls": "three", "B": 700, "K": 1500,
         "N": 1500, "ts": 0, "dp": 2},
        # One training iteration of the paper's MLP, 784-2048-2048-10 at batch 128.
        {"name": "mlp_2048_step", "kind": "mlp", "K0": 784, "H1": 2048, "H2": 2048, "out": 10, "B": 128, "dp": 2},
        # LSTM layer of 1024 units, batch 64, 35 steps; and the paper's width and batch, 1500 units at 20.
        {"name": "lstm_1024", "kind": "lstm", "T": 35, "B": 64, "I": 1024, "H": 1024, "dp": 2},
        {"name": "lstm_1500", "kind": "lstm", "T": 35, "B": 20, "I": 1500, "H": 1500, "dp": 2},
        # Convolution layer (3 x 3 filters, 256 -> 512 channels, 32768 output positions) with rows, or blocks, of its
        # input matrix dropped by predicted sensitivity.
        {"name": "conv_rows", "kind": "conv_rows", "M": 32768, "K": 2304, "N": 512, "run_len": 32},
        {"name": "conv_blocks", "kind": "conv_blocks", "M": 32768, "K": 2304, "N": 512, "ts": 128, "run_len": 32},
    ]


def _size(rng, lo, hi, step):
    """A size spread over the logarithm of lo .. hi, rounded down to a multiple of `step`."""
    return max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))) // step * step)


def draw(rng):
    kind = rng.choice(["row", "row", "row", "tile", "tile", "mlp", "lstm", "lstm", "conv_rows", "conv_blocks"])
    dp = rng.choice([1, 2, 2, 3, 4, 5, 7, 8, 12, 16])
    if kind in ("row", "tile"):
        dtype = rng.choice(["bf16", "bf16", "f32"])
        ts = rng.choice([32, 64, 128]) if kind == "tile" else 0
        odd = kind == "row" and rng.random() < 0.3
        step = ts or (1 if odd else 8)
        # fp32 layers are the small ones; odd sizes belong to layers of up to 2048 units
        top, btop = (4096, 1024) if dtype == "f32" else ((2048, 2048) if odd else (8192, 4096))
        low = max(128, 4 * ts)  # at least 16 tiles: as many units as a distribution has periods
        return {"kind": "layer", "pattern": kind, "dtype": dtype, "calls": rng.choice(["three", "one"]),
                "B": _size(rng, 16, btop, 1 if odd else 4), "K": _size(rng, low, top, step),
                "N": _size(rng, low, top, step), "ts": ts, "dp": dp}
    if kind == "mlp":
        h1, h2 = (_size(rng, 256, 4096, 64) for _ in range(2))
        return {"kind": "mlp", "K0": 784, "H1": h1, "H2": h2, "out": 10, "B": _size(rng, 32, 256, 1), "dp": dp}
    if kind == "lstm":
        step = rng.choice([64, 8, 4])
        I, H = (_size(rng, 128, 1536, step) for _ in range(2))
        return {"kind": "lstm", "T": rng.randint(5, 35), "B": _size(rng, 8, 128, 1), "I": I, "H": H, "dp": dp}
    if kind == "conv_rows":
        return {"kind": "conv_rows", "M": _size(rng, 4096, 32768, 8), "K": 9 * rng.choice([64, 128, 256]),
                "N": rng.choice([64, 128, 256, 512]), "run_len": rng.choice([1, 32])}
    ts = rng.choice([64, 128])
    return {"kind": "conv_blocks", "M": _size(rng, 4096, 32768, ts), "K": 9 * rng.choice([128, 256]),
            "N": rng.choice([64, 128, 256, 512]), "ts": ts, "run_len": rng.choice([1, 32])}


class State:
    """What a training program keeps for one case; the library's objects are given back when it goes."""

    def __init__(self, case):
        self.case, self.it, self.owned, self.ctx = case, 0, [], None
        weakref.finalize(self, State.close, self.owned)

    @staticmethod
    def close(owned):
        for handle, destroy in reversed(owned):
            destroy(handle)

    def open(self, workspace_bytes, dp=None):
        self.ctx = self.own(ard.ard_create(torch.cuda.current_device(), workspace_bytes), ard.ard_destroy)
        if dp is not None:
            K = [0.0] * max(N_PERIODS, dp)
            K[dp - 1] = 1.0
            ard.ard_set_distribution(self.ctx, 0, K)

    def own(self, handle, destroy):
        self.owned.append((handle, destroy))
        return handle


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    s = State(dict(case))
    _PREPARE[case["kind"]](s, s.case, g)
    return s


def run(state):
    return _RUN[state.case["kind"]](state, state.case)


def _randn(g, shape, dtype, scale=1.0):
    return (torch.randn(shape, device="cuda", generator=g) * scale).to(dtype)


# ---- one layer ---------------------------------------------------------------------------------------------
def _prepare_layer(s, c, g):
    B, K, N = c["B"], c["K"], c["N"]
    td = F32 if c["dtype"] == "f32" else BF16
    s.dt = ard.ARD_F32 if c["dtype"] == "f32" else ard.ARD_BF16
    s.open(td.itemsize * B * (N + 8) + 4096, c["dp"])
    kind = ard.ARD_ROW if c["pattern"] == "row" else ard.ARD_TILE
    s.pat = s.own(ard.ard_pattern_create(s.ctx, kind, K, N, c["ts"]), ard.ard_pattern_destroy)
    s.alpha = float(c["dp"])  # 1 / (1 - p)
    s.X, s.dY = _randn(g, (B, K), td), _randn(g, (B, N), td)
    s.W = _randn(g, (N, K), td, K ** -0.5)
    s.Y, s.dX = torch.zeros((B, N), dtype=td, device="cuda"), torch.zeros((B, K), dtype=td, device="cuda")
    s.dW = torch.zeros((N, K), dtype=td, device="cuda")


def _run_layer(s, c):
    B, K, N, dt = c["B"], c["K"], c["N"], s.dt
    ard.ard_sample_pattern(s.ctx, s.pat, 0, SAMPLER_SEED, s.it, 0)
    s.it += 1
    if c["calls"] == "one":
        ard.ard_layer_products(s.ctx, s.pat, dt, dt, B, K, N, s.alpha, s.X, K, s.W, K, s.dY, N, s.Y, N,
                               ard.ARD_OUT_SCATTER_ZEROFILL, s.dX, K, s.dW, K, 1)
    else:
        ard.ard_fwd(s.ctx, s.pat, dt, B, K, N, s.alpha, s.X, K, s.W, K, s.Y, N, ard.ARD_OUT_SCATTER_ZEROFILL)
        ard.ard_bwd_data(s.ctx, s.pat, dt, B, K, N, s.alpha, s.dY, N, 0, s.W, K, s.dX, K)
        ard.ard_bwd_weight(s.ctx, s.pat, dt, dt, B, K, N, s.alpha, s.X, K, s.dY, N, 0, s.dW, K, 1)
    return s.Y, s.dX, s.dW


def _work_layer(c):
    B, K, N, dp = c["B"], c["K"], c["N"], c["dp"]
    es = 4 if c["dtype"] == "f32" else 2
    dy = B * N / dp if c["pattern"] == "row" else B * N
    return {"flops": 3 * 2.0 * B * K * N / dp, "bytes": es * (2.0 * B * K + B * N + dy + K * N / dp + K * N)}


# ---- a stack of layers -------------------------------------------------------------------------------------
def _dims(c):
    return [c["K0"], c["H1"], c["H2"], c["out"]]


def _prepare_mlp(s, c, g):
    B, dims = c["B"], _dims(c)
    s.open(2 * B * max(dims) + 4096, c["dp"])
    s.layers = []
    for l in range(3):
        K, N, hidden = dims[l], dims[l + 1], l < 2
        pat = s.own(ard.ard_pattern_create(s.ctx, ard.ARD_ROW, K, N, 0), ard.ard_pattern_destroy)
        zeros = lambda *shape, dtype=BF16: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
        s.layers.append(dict(
            K=K, N=N, pat=pat, sample=int(hidden), relu=int(hidden), compact_out=int(hidden), dW_is_f32=0,
            alpha=float(c["dp"]) if hidden else 1.0, ldw=K, W=_randn(g, (N, K), BF16, (2.0 / K) ** 0.5),
            bias=_randn(g, (N,), F32, 0.1), Wk=zeros(N, K), A=zeros(B, N), dZ=zeros(B, N), dWk=zeros(N, K),
            dW=zeros(N, K), db=zeros(N, dtype=F32)))
    ard.ard_pattern_set(s.ctx, s.layers[-1]["pat"], 1, 1)
    s.table = ard.mlp_layers(s.layers)
    s.X = torch.rand((B, dims[0]), device="cuda", generator=g).to(BF16)
    s.dOut = _randn(g, (B, dims[-1]), BF16, 1.0 / B)
    s.dX = torch.zeros((B, dims[0]), dtype=BF16, device="cuda")
    s.counter = torch.zeros(1, dtype=torch.int64, device="cuda")  # advanced by the step itself


def _run_mlp(s, c):
    dims = _dims(c)
    ard.ard_mlp_step(s.ctx, s.table, 3, c["B"], s.X, dims[0], s.dOut, dims[-1], s.dX, dims[0], 0, SAMPLER_SEED, 0,
                     s.counter)
    return [s.layers[-1]["A"], s.dX] + [d["dW"] for d in s.layers] + [d["db"] for d in s.layers]


def _work_mlp(c):
    B, dims, dp = c["B"], _dims(c), c["dp"]
    n = [dims[0], dims[1] / dp, dims[2] / dp, dims[3]]
    flops = sum(3 * 2.0 * B * n[l] * n[l + 1] for l in range(3))
    byts = sum(2.0 * n[l] * n[l + 1] + 2.0 * dims[l] * dims[l + 1] + 4 * dims[l + 1] for l in range(3))
    return {"flops": flops, "bytes": byts + 2.0 * B * (2 * dims[0] + 2 * dims[3])}


# ---- an LSTM layer -----------------------------------------------------------------------------------------
def _prepare_lstm(s, c, g):
    T, B, I, H = c["T"], c["B"], c["I"], c["H"]
    s.open(2 * B * (I + H) * 4 + 4096, c["dp"])
    s.pat = s.own(ard.ard_pattern_create(s.ctx, ard.ARD_ROW, I + H, H, 0), ard.ard_pattern_destroy)
    W = ((torch.rand((4 * H, I + H), device="cuda", generator=g) * 2 - 1) * 0.03).to(BF16)
    s.layer = lstm.LstmLayer(s.ctx, s.pat, T, B, I, H, W)
    s.X, s.dH = _randn(g, (T, B, I), BF16), _randn(g, (T, B, H), F32, 1.0 / 64)


def _run_lstm(s, c):
    ard.ard_sample_pattern(s.ctx, s.pat, 0, SAMPLER_SEED, s.it, 0)
    s.it += 1
    s.layer.load_inputs(s.X)
    h = s.layer.forward(float(c["dp"]))
    dx, dw = s.layer.backward(float(c["dp"]), s.dH)
    return h, dx, dw


def _work_lstm(c):
    T, B, I, H, n = c["T"], c["B"], c["I"], c["H"], c["H"] / c["dp"]
    return {"flops": 3 * 2.0 * T * B * (I + n) * 4 * n,
            "bytes": 2.0 * T * B * (I + H) + 4.0 * T * B * (n + I) + 2.0 * 4 * n * (I + n) + 4.0 * 4 * H * (I + H)}


# ---- a convolution layer's input matrix ----------------------------------------------------------------------
REGION_ROWS, K_FRAC, T_FRAC, THRESHOLD, M_PROB, N_PROB, CAP_OF_18 = 8, 0.05, 0.3, 0.5, 0.2, 0.8, 6


def _conv_tensors(s, c, g, level):
    M, K, N = c["M"], c["K"], c["N"]
    # post-ReLU input with quiet and busy regions, so that both kinds of region occur
    s.A = (torch.relu(torch.randn((M, K), device="cuda", generator=g)) * level).to(BF16)
    s.W = _randn(g, (N, K), BF16, K ** -0.5)
    s.dA, s.dW = torch.zeros((M, K), dtype=BF16, device="cuda"), torch.zeros((N, K), dtype=BF16, device="cuda")
    s.open(4096)


def _levels(g, shape):
    return torch.tensor([0.1, 1.0, 4.0], device="cuda")[torch.randint(0, 3, shape, device="cuda", generator=g)]


def _prepare_conv_rows(s, c, g):
    M, K, N = c["M"], c["K"], c["N"]
    _conv_tensors(s, c, g, _levels(g, (M // REGION_ROWS,)).repeat_interleave(REGION_ROWS)[:, None])
    s.rows = s.own(ard.ard_rows_create(s.ctx, M, REGION_ROWS), ard.ard_rows_destroy)
    s.dY, s.Y = _randn(g, (M, N), BF16), torch.zeros((M, N), dtype=BF16, device="cuda")
    cap = (M + 63) // 64 * 64
    s.Ak = torch.zeros((cap, K), dtype=BF16, device="cuda")
    s.dYk = torch.zeros((cap, N), dtype=BF16, device="cuda")


def _run_conv_rows(s, c):
    M, K, N = c["M"], c["K"], c["N"]
    ard.ard_sensitivity_predict(s.ctx, s.rows, ard.ARD_BF16, s.A, K, K, K_FRAC, c["run_len"], T_FRAC, THRESHOLD, M_PROB,
                                N_PROB, SAMPLER_SEED, s.it, 0)
    ard.ard_rows_sample(s.ctx, s.rows, SAMPLER_SEED, s.it, 0)
    s.it += 1
    ard.ard_rows_products(s.ctx, s.rows, ard.ARD_BF16, M, K, N, 1.0, s.A, K, s.W, K, s.dY, N, s.Ak, K, s.dYk, N, s.Y, N,
                          s.dA, K, s.dW, K)
    return s.Y, s.dA, s.dW


def _prepare_conv_blocks(s, c, g):
    M, K, N, ts = c["M"], c["K"], c["N"], c["ts"]
    _conv_tensors(s, c, g, _levels(g, (M // ts, K // ts)).repeat_interleave(ts, 0).repeat_interleave(ts, 1))
    s.blocks = s.own(ard.ard_blocks_create(s.ctx, M, K, ts), ard.ard_blocks_destroy)
    s.dY, s.Y = _randn(g, (N, M), BF16), torch.zeros((N, M), dtype=BF16, device="cuda")  # one row per channel


def _run_conv_blocks(s, c):
    M, K, N = c["M"], c["K"], c["N"]
    cap = max(1, CAP_OF_18 * (K // c["ts"]) // 18)
    ard.ard_blocks_predict(s.ctx, s.blocks, ard.ARD_BF16, s.A, K, K_FRAC, c["run_len"], T_FRAC, THRESHOLD, cap,
                           SAMPLER_SEED, s.it, 0)
    ard.ard_blocks_sample(s.ctx, s.blocks, M_PROB, N_PROB, SAMPLER_SEED, s.it, 0)
    s.it += 1
    ard.ard_blocks_products(s.ctx, s.blocks, ard.ARD_BF16, N, 1.0, s.A, K, s.W, K, s.dY, M, s.Y, M, s.dW, K, s.dA, K, 1)
    return s.Y, s.dA, s.dW


def _work_conv(c):
    M, K, N = c["M"], c["K"], c["N"]
    # kept share: 54 % of the rows; of the blocks, a third sensitive at 80 % and the rest at 20 %
    f = 0.54 if c["kind"] == "conv_rows" else 0.4
    kept_dy = M * N * (f if c["kind"] == "conv_rows" else 1.0)
    return {"flops": 3 * 2.0 * f * M * K * N, "bytes": 2.0 * (f * M * K + M * K + M * N + kept_dy + 2 * N * K)}


_PREPARE = {"layer": _prepare_layer, "mlp": _prepare_mlp, "lstm": _prepare_lstm, "conv_rows": _prepare_conv_rows,
            "conv_blocks": _prepare_conv_blocks}
_RUN = {"layer": _run_layer, "mlp": _run_mlp, "lstm": _run_lstm, "conv_rows": _run_conv_rows,
        "conv_blocks": _run_conv_blocks}
_WORK = {"layer": _work_layer, "mlp": _work_mlp, "lstm": _work_lstm, "conv_rows": _work_conv, "conv_blocks": _work_conv}


def work(case):
    return _WORK[case["kind"]](case)


def tolerance(case):
    # About four times what the results differ by from fp64 references, or from the same work with its sums in another
    # order: 8e-7 for fp32 layers of a fan-in of 2048; 1.7e-3, the rounding of the outputs, for bf16 ones.
    if case.get("dtype") == "f32":
        return {"rel": 4e-6, "max": 3e-5}
    # Chains with bf16 activations or gate gradients in between measured 8e-4 (LSTM) and 4e-4 (MLP); the largest single
    # difference there comes from an activation whose sum is within rounding of zero and switches its gradient.
    return {"rel": 5e-3, "max": {"mlp": 0.5, "lstm": 0.1}.get(case["kind"], 5e-2)}
