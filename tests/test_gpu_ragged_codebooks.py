"""bf16 engines whose codebooks do not add up to whole 32-column blocks of the LM head's product."""
import numpy as np
import pytest
import torch

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case, check_levels, check_walk_against_trace, tolerance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [(16, 16, 16, 16),      # 48 columns: a block and a half
                               (9, 11, 5, 7),         # 23: rows that start off the 16-byte boundaries
                               (40, 100, 61),         # 161: one more than five blocks
                               (3, 31), (200, 33, 64)])
@pytest.mark.parametrize("batch,beam", [(2, 5),       # every product streams its weights
                                        (40, 9)])     # the general kernel
def test_ragged_codebooks_match_the_oracle(T, batch, beam):
    n = min(3_000, int(np.prod(T)) // 3)
    rng = np.random.default_rng(len(T) + batch)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=2, L=len(T), T=T, n_items=n, batch=batch, beam=beam, n_hist=9)
    torch.cuda.empty_cache()
    dirt = torch.full((1 << 28,), float("nan"), device="cuda")             # what the arena is likely to find
    torch.cuda.synchronize()
    del dirt
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n, size=(batch, 9))]).prefill()
    out = case.eng.decode(beam, mode=binding.MODE_VERIFIED, trace=True)
    ar = case.eng.decode(beam, mode=binding.MODE_AR)
    assert torch.equal(out["codes"], ar["codes"]) and torch.equal(out["count"], ar["count"])
    check_walk_against_trace(out, w.batch, w.L)
    beams, scores = out["trace"]["beams"].cpu().numpy(), out["trace"]["beam_scores"].cpu().numpy()
    for b in (0, batch // 2, batch - 1):
        check_levels(case, b, beams[:, b], scores[:, b], beam, tol=tolerance(w))
    case.eng.close()


@pytest.mark.parametrize("T", [(8, 20, 300),           # a level of one code a lane in the form of 16
                               (8, 600, 20),           # ... and of 32, whose blocks have at most 8 warps, behind a wider level
                               (16, 20, 300, 40), (7, 513, 33, 512)])
@pytest.mark.parametrize("dtype,batch,beam", [("fp32", 2, 5), ("bf16", 3, 9), ("bf16", 2, 20)])
@pytest.mark.parametrize("final_mask", [0, 1])         # the last level's mask by hash probes, or from the prefix map
def test_levels_on_different_sides_of_the_code_limits(T, dtype, batch, beam, final_mask):
    """One launch selects level after level in the form of the widest: every level against the oracle, the whole walk with the true
    beams as the draft tree, and with the head's own tree."""
    L, n = len(T), 3_000
    rng = np.random.default_rng(L + beam)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["tiny" if dtype == "fp32" else "small"], n_layers=1, L=L, T=T, n_items=n, batch=batch, beam=beam, n_hist=5)
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n, size=(batch, 5))]).prefill()
    case.eng.set_option(binding.OPT_FINAL_MASK, final_mask)
    ar = case.eng.decode(beam, mode=binding.MODE_AR, trace=True)
    tree = ar["trace"]["beams"].clone()
    sizes = (tree[:, :, :, 0] >= 0).sum(dim=2).to(torch.int32).contiguous()
    accepted = case.eng.decode_with_draft_tree(beam, tree, sizes, trace=True)
    natural = case.eng.decode(beam, mode=binding.MODE_VERIFIED, trace=True)
    assert accepted["stats"].rounds == 1
    for out in (accepted, natural):
        assert torch.equal(out["codes"], ar["codes"]) and torch.equal(out["count"], ar["count"])
        assert torch.equal(out["trace"]["beams"], ar["trace"]["beams"])
        check_walk_against_trace(out, batch, L)
    scores = ar["trace"]["beam_scores"].cpu().numpy()
    for b in range(batch):
        check_levels(case, b, tree[:, b].cpu().numpy(), scores[:, b], beam, tol=tolerance(w))
    case.eng.close()
