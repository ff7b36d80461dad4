"""Stacked LSTM layers off the 16-byte grid: the recurrences run from pre-activations and hand back a second copy of their gate
gradients in the caller's layout, both layers against the oracle."""
import pytest

from paper_2203_05705_b200 import ard
from gpu_helpers import TOL
from test_gpu_lstm_stack import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B,dims,dps", [(4, 20, (52, 204, 100), ((2, 2), (3, 1))), (3, 33, (57, 131, 98), ((1, 1), (5, 4))),
                                          (2, 70, (64, 1196, 36), ((4, 1), (1, 1)))])
def test_two_layers_off_the_grid(T, B, dims, dps):
    errs = _run(T, B, dims, dps, (1.5, 2.0), T + B)
    assert max(errs.values()) <= TOL[ard.ARD_BF16], errs
