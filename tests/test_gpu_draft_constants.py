"""The draft head's per-request constants W_logit_l h_l: of few requests one product for all levels, of many a product per level."""
import ctypes
import math

import numpy as np
import pytest
import torch

from gpu_helpers import Case
from paper_2511_18793_b200 import binding, synth


def _arena(T, batch):
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, d_model=64, n_q_heads=1, n_kv_heads=1, d_ffn=64, L=len(T), T=T, n_items=1_000, batch=batch,
                     beam=1, n_hist=1)
    return binding.lib.nezha_arena_bytes(ctypes.byref(binding.make_config(w)), w.n_items, w.load_factor)


@pytest.mark.parametrize("T", [(1024,) * 6, (256,) * 4])
def test_many_requests_constants_take_a_row_per_level(T):
    """A request more in a large engine does not cost another (L + 1) sum(T) constants, only its own L max(T)."""
    L, each = len(T), (_arena(T, 2_048) - _arena(T, 1_024)) / 1_024
    # what else grows with the codes: the LM head's logits of a pass, B_1's and the draft head's (three buffers); and 24 KB for all the rest
    logits = 4 * ((L + 1) * (sum(T[1:]) + 31) + T[0] + 3 * max(T))
    assert each < logits + 4 * L * max(T) + 24 * 1024, (each, logits)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [(256,) * 4, (40, 100, 61)])
def test_constants_of_both_forms_agree(T):
    n = min(3_000, math.prod(T) // 3)
    rng = np.random.default_rng(len(T))
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, L=len(T), T=T, n_items=n, batch=257, beam=3, n_hist=2)
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n, size=(257, 2))]).prefill()        # per level

    def results(batch):
        logits = []
        for level in range(w.L):
            pre = torch.from_numpy(np.stack([cat[rng2.integers(0, n, size=w.beam), :level] for _ in range(257)])).cuda()[:batch].contiguous()
            logits.append(case.eng.draft_logits(w.beam, level, pre if level else None).clone())
        out = case.eng.decode(w.beam, mode=binding.MODE_DRAFT)
        case.eng.sync()
        return logits, out["codes"].clone(), out["scores"].clone()

    rng2 = np.random.default_rng(1)
    many, many_codes, many_scores = results(257)
    case.eng.prefill(case.hist_dev[:256].contiguous(), case.n_hist[:256].contiguous())        # at once
    rng2 = np.random.default_rng(1)
    few, few_codes, few_scores = results(256)
    for a, b in zip(many, few):
        # the same bf16 operands, fp32 sums of 512 products of about 0.02 in another order at most
        assert (a[:256] - b).abs().max().item() < 1e-5
    assert torch.allclose(many_scores[:256], few_scores, atol=1e-4)
    model, head, _ = case.oracle
    for b in (0, 255, 256):
        h = case.req(b).h
        ref = head.logits(0, h[1], h[0])
        assert np.abs(many[0][b, 0].cpu().numpy() - ref).max() < 2e-2
    case.eng.close()
