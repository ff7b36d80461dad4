"""What the LSTM layer hands to the native library: the kernels read [T][B][H] floats behind a bare pointer, so anything
that is not that is refused before the call, and a gradient of another type or order is brought into it."""
import pytest
import torch

from paper_2203_05705_b200 import ard
from paper_2203_05705_b200.lstm import LstmLayer

T, B, I, H = 3, 4, 5, 6


@pytest.fixture
def layer(monkeypatch):
    ly = object.__new__(LstmLayer)       # the buffers on the CPU: no call reaches the library
    ly.ctx = ly.pat = None
    ly.T, ly.B, ly.I, ly.H, ly.KH = T, B, I, H, I + H
    z = lambda *s: torch.zeros(*s)       # noqa: E731
    ly.XH, ly.W, ly.C, ly.G, ly.Z = z(T + 1, B, I + H), z(4 * H, I + H), z(T + 1, B, H), z(T, B, 4 * H), z(B, 4 * H)
    ly.DZ, ly.D, ly.dc, ly.dW = z(T, B, 4 * H), z(T, B, I + H), z(B, H), z(4 * H, I + H)
    ly.calls = []
    monkeypatch.setattr(ard, "ard_lstm_backward_dh", lambda *a: ly.calls.append(a))
    return ly


@pytest.mark.parametrize("shape", [(T - 1, B, H), (T, B - 1, H), (T, B, H - 1), (T, 1, H), (1, B, H), (T, B), (T * B * H,),
                                   (T + 1, B, H), (T, B, H, 1)])
def test_a_gradient_of_another_shape_is_refused(layer, shape):
    with pytest.raises((ValueError, RuntimeError)):
        layer.backward(1.0, torch.zeros(shape))
    assert layer.calls == []


def test_a_gradient_on_another_device_is_refused(layer):
    with pytest.raises((ValueError, RuntimeError)):
        layer.backward(1.0, torch.zeros((T, B, H), device="meta"))
    assert layer.calls == []


@pytest.mark.parametrize("make", [lambda g: g, lambda g: g.to(torch.bfloat16), lambda g: g.double(),
                                  lambda g: g.transpose(0, 2).contiguous().transpose(0, 2), lambda g: g[:1].expand(T, B, H)])
def test_types_and_orders_are_brought_into_the_kernels_form(layer, make):
    dH = make(torch.randn(T, B, H))
    dX, dW = layer.backward(1.0, dH)
    (call,) = layer.calls
    handed = [a for a in call if isinstance(a, torch.Tensor) and tuple(a.shape) == (T, B, H)]
    assert len(handed) == 1 and handed[0].dtype == torch.float32 and handed[0].is_contiguous()
    assert torch.equal(handed[0], dH.to(torch.float32))
    assert tuple(dX.shape) == (T, B, I) and dW is layer.dW
