"""The K best of the per-beam lists where scores tie: by score, then the parent's rank, then the code -- for one candidate up to more
than are compared all with all (1,024), beams that are fewer or more than K, and codebooks smaller than K."""
import numpy as np
import pytest
import torch

from gpu_helpers import Case
from paper_2511_18793_b200 import synth

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
