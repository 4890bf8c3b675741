"""fp32 engines whose layers run their norms, rotary embedding and SwiGLU inside the products, and engines just outside that, against the
fp64 oracle: head sizes 16 to 128, grouped heads, ragged codebooks and feed-forward widths, one row to several tiles of rows."""
import numpy as np
import pytest
import torch

from gpu_helpers import Case, tolerance
from paper_2511_18793_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,Hq,Hkv,F,T,batch,n_hist", [
    (64, 4, 4, 256, (32, 32, 32), 4, 20), (32, 2, 1, 7, (9, 11, 5), 1, 1), (64, 2, 1, 100, (9, 31, 100), 3, 9),
    (128, 2, 2, 36, (33, 17, 8), 2, 5), (256, 2, 1, 260, (32, 32, 32), 1, 11), (272, 17, 1, 64, (32, 32, 32), 2, 3)])
def test_narrow_fp32_layers(d, Hq, Hkv, F, T, batch, n_hist):
    w = synth.scaled(synth.WORKLOADS["tiny"], d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, d_ffn=F, T=T, n_items=200, batch=batch, n_hist=n_hist)
    case = Case(w).prefill()
    h = case.eng.get_hidden().cpu().numpy()
    model = case.oracle[0]
    rng = np.random.default_rng(d)
    pre = np.stack([rng.integers(0, t, size=(batch, w.beam)) for t in T[:2]], axis=2).astype(np.int32)
    got = case.eng.primary_logits(w.beam, 2, torch.from_numpy(pre).cuda()).cpu().numpy()
    for b in range(batch):
        assert np.abs(h[b] - case.req(b).h).max() < 2e-5
        ref = model.next_level_logits_many(case.req(b), [tuple(p) for p in pre[b]])
        assert np.abs(got[b] - np.stack(ref)).max() < tolerance(w)
    case.eng.close()
