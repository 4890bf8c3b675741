"""The draft head's per-request constants W_logit_l h_l: one product for all levels while it is small, else a product per level."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_helpers import Case
from paper_2511_18793_b200 import binding, synth


def _arena(T, batch):
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, d_model=64, n_q_heads=1, n_kv_heads=1, d_ffn=64, L=len(T), T=T, n_items=1_000, batch=batch,
                     beam=1, n_hist=1)
    return binding.lib.nezha_arena_bytes(ctypes.byref(binding.make_config(w)), w.n_items, w.load_factor)


def test_many_requests_constants_take_a_row_per_level():
    """A request more in a large engine does not cost another (L + 1) sum(T) constants, only its own L max(T)."""
    T, batch = (1024,) * 6, 4_096
    L, each = len(T), (_arena(T, 2 * batch) - _arena(T, batch)) / batch
    # what else grows with the codes: the LM head's logits of a pass, B_1's and the draft head's (three buffers); and 24 KB for all the rest
    logits = 4 * ((L + 1) * (sum(T[1:]) + 31) + T[0] + 3 * max(T))
    assert each < logits + 4 * L * max(T) + 24 * 1024, (each, logits)


@pytest.mark.gpu
@pytest.mark.parametrize("T,batch,few", [((1024,) * 4, 763, 762),        # 16.002 and 15.98 GFLOP: a product per level, and one product
                                         ((1000,) * 3, 800, 100)])       # no multiple of 32 codes: one product for both
def test_constants_of_both_forms_agree(T, batch, few):
    n = 3_000
    rng = np.random.default_rng(len(T))
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, L=len(T), T=T, n_items=n, batch=batch, beam=3, n_hist=2)
    case = Case(w, catalog=cat, hist=cat[rng.integers(0, n, size=(batch, 2))])
    case.eng.set_option(binding.OPT_DRAFT_FILTER, 0)         # (every drafted tuple is returned)
    pre = [torch.from_numpy(cat[rng.integers(0, n, size=(batch, w.beam)), :level]).cuda() for level in range(w.L)]

    def results(k):
        case.eng.prefill(case.hist_dev[:k].contiguous(), case.n_hist[:k].contiguous())
        logits = [case.eng.draft_logits(w.beam, level, pre[level][:k].contiguous() if level else None).clone() for level in range(w.L)]
        out = case.eng.decode(w.beam, mode=binding.MODE_DRAFT)
        case.eng.sync()
        return logits, out["scores"].clone()

    many, many_scores = results(batch)
    fewer, few_scores = results(few)
    for a, b in zip(many, fewer):
        # the same bf16 operands, fp32 sums of 512 products of about 0.02 in another order at most
        assert (a[:few] - b).abs().max().item() < 1e-5
    assert torch.isfinite(few_scores).all() and (many_scores[:few] - few_scores).abs().max().item() < 1e-4
    head = case.oracle[1]
    for b in (0, few - 1, batch - 1):
        h = case.req(b).h
        assert np.abs(many[0][b, 0].cpu().numpy() - head.logits(0, h[1], h[0])).max() < 2e-2
    case.eng.close()
