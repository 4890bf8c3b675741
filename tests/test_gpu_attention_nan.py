"""Attention over keys that are not numbers: the result is not a number, as the softmax over them is not one."""
import pytest
import torch

from paper_2511_18793_b200 import synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


def test_a_lane_group_that_sees_only_nan_scores_spoils_the_result():
    # four levels: the first codes of the items stand at the positions 1, 5, 9, 13, all of one lane group's first step
    w = synth.scaled(synth.WORKLOADS["tiny"], n_layers=1, L=4, T=(32,) * 4, batch=2, n_hist=4)
    weights = synth.make_weights(w, device="cuda")
    weights["embed"][: w.T[0]] = float("nan")
    case = Case(w, weights=weights).prefill()
    assert torch.isnan(case.eng.get_hidden()).all().item()
    case.eng.close()
