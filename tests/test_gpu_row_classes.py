"""Engines whose passes have more than 128 rows stream the weights of the products for which that pays, by a rule on the
product and the engine's largest pass: both decode modes must still agree item for item at every size."""
import pytest
import torch

from paper_2511_18793_b200 import synth
from gpu_helpers import Case, check_levels, check_walk_against_trace, wide_tolerance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,beam,n_hist", [(13, 10, 12),      # 260 rows: three row tiles, the last nearly empty
                                               (32, 10, 12),      # 640: the largest class
                                               (33, 10, 12),      # 660: none
                                               (2, 10, 60)])      # 40 rows; a prompt chunk of 368 tokens in three row tiles
def test_modes_agree_in_every_row_class(batch, beam, n_hist):
    w = synth.scaled(synth.WORKLOADS["paper"], n_layers=2, batch=batch, beam=beam, n_hist=n_hist)
    case = Case(w).prefill()
    out = case.eng.decode(w.beam, mode=1, trace=True)
    ar = case.eng.decode(w.beam, mode=2)
    for k in ("codes", "count"):           # (the scores to the attention's choice of kernel, which goes by the rows of a pass)
        assert torch.equal(out[k], ar[k]), k
    check_walk_against_trace(out, w.batch, w.L)
    beams, scores = out["trace"]["beams"].cpu().numpy(), out["trace"]["beam_scores"].cpu().numpy()
    for b in {0, batch - 1}:
        check_levels(case, b, beams[:, b], scores[:, b], w.beam, tol=wide_tolerance(w))
    case.eng.close()
