"""The whole-sequence kernels over the whole grid where the device has no room for clusters of CTAs: patterns that the clusters would take
run in them, down to the forms for few kept units (four units a CTA, BPTT without the exchange).  The tests of these kernels, with the
launches in clusters refused."""
import pytest

import test_gpu_lstm_persistent as persistent
import test_gpu_lstm_shapes as shapes
from paper_2203_05705_b200 import ard
from gpu_helpers import Ctx

pytestmark = pytest.mark.gpu


class GridWideCtx(Ctx):
    def __init__(self, *args):
        super().__init__(*args)
        ard.ard_set_option(self.h, ard.ARD_OPT_LSTM_REFUSE, 1)


@pytest.fixture(autouse=True)
def grid_wide(monkeypatch):
    monkeypatch.setattr(persistent, "Ctx", GridWideCtx)
    monkeypatch.setattr(shapes, "Ctx", GridWideCtx)


@pytest.mark.parametrize("T,B,I,H", [(6, 33, 128, 264), (3, 1, 64, 1024)])
def test_forward(T, B, I, H):
    persistent.test_persistent_forward_matches_the_oracle_and_the_per_step_path(T, B, I, H)


def test_both_forms_of_the_forward_recurrence():
    persistent.test_compact_recurrence_and_full_width_recurrence_agree()


@pytest.mark.parametrize("T,B,I,H", [(5, 33, 128, 264), (3, 128, 64, 128), (4, 7, 192, 1024)])
def test_bptt(T, B, I, H):
    persistent.test_persistent_bptt_matches_the_oracle_and_the_per_step_path(T, B, I, H)


@pytest.mark.parametrize("T,B,I,H,periods", [(4, 70, 64, 520, [(2, 2), (5, 1), (9, 4)]), (3, 64, 128, 1024, [(4, 3), (7, 7), (16, 2)])])
def test_both_forms_of_the_bptt_recurrence(T, B, I, H, periods):
    persistent.test_both_forms_of_the_bptt_recurrence_match_the_oracle(T, B, I, H, periods)


def test_replays_that_need_two_launches_over_the_grid():
    persistent.test_a_sequence_replays_from_a_cuda_graph_with_a_new_pattern_each_time()


@pytest.mark.parametrize("T,B,I,H", [(4, 20, 52, 204), (3, 33, 57, 131), (3, 70, 36, 1100), (3, 20, 300, 1500)])
def test_any_shape(T, B, I, H):
    shapes.test_any_shape_matches_the_oracle(T, B, I, H, 1)
