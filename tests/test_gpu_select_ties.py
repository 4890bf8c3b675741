"""The K best of the per-beam lists where scores tie: by score, then the parent's rank, then the code -- for one candidate up to more
than are compared all with all (1,024), beams that are fewer or more than K, and codebooks smaller than K; also where the ties come of
the rounding of a beam's score plus a code's log-probability, and a beam's list was made before the sum."""
import numpy as np
import pytest
import torch

from gpu_helpers import Case, assert_topk_matches, check_levels, tolerance
from oracle import nezha_oracle as O
from paper_2511_18793_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return Case(synth.scaled(synth.WORKLOADS["tiny"], T=(7, 256, 600), n_items=200, n_layers=1, batch=1, n_hist=1, beam=128), max_beam=128)


@pytest.mark.parametrize("n_beams,K", [(1, 1), (1, 40), (3, 1), (3, 5), (10, 10), (20, 20), (32, 32), (33, 33), (40, 7), (5, 128), (128, 128)])
@pytest.mark.parametrize("level", [0, 1, 2])
def test_ties_go_by_parent_then_code(ctx, n_beams, K, level):
    T = ctx.w.T[level]
    rng = np.random.default_rng(n_beams * 1000 + K * 3 + level)
    base = -0.25 * rng.integers(0, max(2, n_beams // 3), size=n_beams)         # few distinct scores, exact in binary
    codes = np.zeros((1, n_beams, ctx.w.L), dtype=np.int32)
    parent, code, score, count = ctx.eng.select(
        torch.zeros(1, n_beams, T, device="cuda"), torch.from_numpy(base.astype(np.float32))[None].cuda(),
        torch.from_numpy(codes).cuda() if level else None, torch.tensor([n_beams], dtype=torch.int32, device="cuda"), K, level, T, False)
    want = sorted((-b, r, t) for r, b in enumerate(base) for t in range(T))[:K]
    n = len(want)
    assert int(count) == n
    assert parent[0, :n].tolist() == [r for _, r, _ in want] and code[0, :n].tolist() == [t for _, _, t in want]
    assert (parent[0, n:] == -1).all() and torch.isinf(score[0, n:]).all()
    lp = np.array([-s for s, _, _ in want]) - np.log(T)
    assert np.abs(score[0, :n].cpu().numpy() - lp).max() < 1e-5                # fp32 sums of at most 600 equal terms


def _rounded_sums(eng, logits, base, K, level, n_live):
    """What nezha_select returns for per_beam = K < T.  The K best codes of a beam and their log-probabilities are those of a call of its
    own, where the beam's score is 0 and nothing is rounded; the sums are rounded as fp32 sums are, whatever adds them."""
    n, T = logits.shape
    codes = torch.zeros(n, 1, level, dtype=torch.int32, device="cuda")
    _, code, lp, count = eng.select(logits[:, None].contiguous(), torch.zeros(n, 1, device="cuda"), codes,
                                    torch.ones(n, dtype=torch.int32, device="cuda"), K, level, K, False)
    code, lp, count = code.cpu().numpy(), lp.cpu().numpy(), count.cpu().numpy()
    cands = [(-(np.float32(base[r]) + lp[r, i]), r, int(code[r, i])) for r in range(n_live) for i in range(count[r])]
    ties = sum(base[r] + lp[r, i] == base[r] + lp[r, i + 1] and code[r, i] > code[r, i + 1] for r in range(n_live) for i in range(count[r] - 1))
    return sorted(cands)[:K], int(ties)


@pytest.fixture(scope="module")
def many():
    """As ctx, for 128 requests."""
    return Case(synth.scaled(synth.WORKLOADS["tiny"], T=(7, 256, 600), n_items=200, n_layers=1, batch=128, n_hist=1, beam=128), max_beam=128)


@pytest.mark.parametrize("n_beams,n_live,K", [(1, 1, 2), (1, 1, 10), (1, 1, 128), (2, 2, 2), (2, 2, 10), (3, 3, 10), (3, 2, 128), (10, 3, 10),
                                              (10, 10, 10), (128, 5, 128),
                                              (40, 40, 40), (128, 128, 100)])          # (more than 1,024 stay in the running)
@pytest.mark.parametrize("base", [-20.0, -1000.0])
@pytest.mark.parametrize("level", [1, 2])
def test_sums_that_round_to_the_same_score(many, n_beams, n_live, K, base, level):
    T = many.w.T[level]
    rng = np.random.default_rng(n_beams * 1000 + K * 3 + level)
    # groups of codes a few units in the last place apart: distinct log-probabilities, whose sums with a score of 20 or 1,000 are not
    z = (rng.integers(0, 40, size=(n_beams, T)) / 10 + rng.integers(0, 5, size=(n_beams, T)) * 2.0 ** -21).astype(np.float32)
    score = (base - 0.25 * rng.integers(0, 3, size=n_beams)).astype(np.float32)
    if n_live >= 40:
        score[n_live - 1] = base - 4_000                   # one beam far behind: nothing of the others' lists is worse than its best
    logits = torch.from_numpy(z).cuda()
    want, ties = _rounded_sums(many.eng, logits, score, K, level, n_live)
    assert ties > 0 or K == 2                                # (the lists do hold pairs whose order the sum decides)
    codes = torch.zeros(1, n_beams, level, dtype=torch.int32, device="cuda")
    parent, code, got, count = many.eng.select(logits[None], torch.from_numpy(score).cuda()[None], codes,
                                               torch.tensor([n_live], dtype=torch.int32, device="cuda"), K, level, K, False)
    assert int(count) == len(want) == K
    assert parent[0].tolist() == [r for _, r, _ in want] and code[0].tolist() == [t for _, _, t in want]
    assert got[0].tolist() == [-s for s, _, _ in want]


@pytest.mark.parametrize("T,n_items,level_filter", [((32, 32, 32), 6, 1), ((3, 32, 32), 400, 0), ((3, 32, 32), 7, 1)])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_drafting_from_fewer_beams_than_are_kept(T, n_items, level_filter, dtype):
    """A thin catalogue with the filter at every level, a first codebook smaller than the beam, and both."""
    w = synth.scaled(synth.WORKLOADS["tiny" if dtype == "fp32" else "small"], L=3, T=T, n_items=n_items, n_layers=1, batch=3, beam=9, n_hist=4)
    rng = np.random.default_rng(n_items)
    cat = np.stack([rng.integers(0, t, size=n_items) for t in T], axis=1).astype(np.int32)
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n_items, size=(3, 4))]).prefill()
    case.eng.set_option(binding.OPT_LEVEL_FILTER, level_filter)
    model, head, V = case.oracle
    draft = {k: v.cpu().numpy() for k, v in case.eng.decode(w.beam, mode=binding.MODE_DRAFT).items() if k in ("codes", "scores", "count")}
    out, ar = case.eng.decode(w.beam, mode=binding.MODE_VERIFIED, trace=True), case.eng.decode(w.beam, mode=binding.MODE_AR)
    assert torch.equal(out["codes"], ar["codes"]) and torch.equal(out["count"], ar["count"])
    beams, scores = out["trace"]["beams"].cpu().numpy(), out["trace"]["beam_scores"].cpu().numpy()
    for b in range(w.batch):
        check_levels(case, b, beams[:, b], scores[:, b], w.beam, every_level=bool(level_filter))
        if dtype == "fp32":
            ref = O.nezha_draft(head, case.req(b), w.beam, V, every_level=bool(level_filter))[-1]
            assert_topk_matches(draft["codes"][b], draft["scores"][b], draft["count"][b], ref, w.beam, tolerance(w))
        assert V.contains(draft["codes"][b, : draft["count"][b]]).all()
    case.eng.close()
