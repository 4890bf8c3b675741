"""nezha_select with the filter at an earlier level and beam codes that the caller did not check."""
import numpy as np
import pytest
import torch

from paper_2511_18793_b200 import synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,level", [((32,) * 4, 2), ((32,) * 4, 1), ((200, 70, 6), 1)])      # bit sets of one and of four words
def test_a_beam_outside_the_code_space_has_no_valid_extension(T, level):
    w = synth.scaled(synth.WORKLOADS["tiny"], L=len(T), T=T, n_items=5_000, batch=2, beam=5, n_hist=1)
    rng = np.random.default_rng(level)
    cat = np.stack([rng.integers(0, t, size=w.n_items) for t in T], axis=1).astype(np.int32)
    case = Case(w, catalog=cat, hist=cat[:2, None])
    bad = [[2 ** 31 - 1] * level, [-1] * level, [0] * (level - 1) + [T[level - 1]]]      # keys of 2^31 and more, of 2^64 - 1, one past the last
    n_beams = 5
    codes = torch.tensor(np.stack([np.stack([cat[0, :level], bad[0], cat[1, :level], bad[1], bad[2]]),
                                   np.stack([bad[2], bad[1], bad[0], cat[2, :level], cat[3, :level]])]), dtype=torch.int32, device="cuda")
    good = torch.tensor([[0, 2], [3, 4]], device="cuda")
    g = torch.Generator(device="cuda").manual_seed(5)
    logits = torch.randn(2, n_beams, T[level], device="cuda", generator=g)
    scores = torch.zeros(2, n_beams, device="cuda")
    live = torch.full((2,), n_beams, dtype=torch.int32, device="cuda")
    parent, code, score, count = case.eng.select(logits, scores, codes, live, w.beam, level, T[level], True)
    rows = torch.arange(2, device="cuda")[:, None]
    only = case.eng.select(logits[rows, good].contiguous(), scores[:, :2].contiguous(), codes[rows, good].contiguous(),
                           torch.full((2,), 2, dtype=torch.int32, device="cuda"), w.beam, level, T[level], True)
    case.eng.sync()
    mapped = torch.where(only[0] >= 0, good.gather(1, only[0].clamp(min=0).long()).int(), only[0])
    assert torch.equal(parent, mapped) and torch.equal(code, only[1]) and torch.equal(score, only[2]) and torch.equal(count, only[3])
    assert (count > 0).all().item()
    case.eng.close()
