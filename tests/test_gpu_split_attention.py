"""Attention of a few requests over long contexts: the tiles split over the CTAs of a cluster."""
import json

import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2511_18793_b200 import synth
from gpu_helpers import Case, check_levels, check_walk_against_trace, hidden_tolerance, tolerance

pytestmark = pytest.mark.gpu


def _attention_launches(call, path):
    """The call's result, and (kernel, grid) of the attention launches that it makes (None where another profiler holds the process)."""
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        torch.zeros(1, device="cuda")
        out = call()
        torch.cuda.synchronize()
    p.export_chrome_trace(str(path))
    kernels = [(e["name"], e["args"]["grid"]) for e in json.loads(path.read_text())["traceEvents"] if e.get("cat") == "kernel"]
    return out, [k for k in kernels if "attn" in k[0]] if kernels else None


@pytest.mark.parametrize("heads,kv_heads,lens,beam,split", [
    (4, 2, (400,), 5, 8),            # hd 128, 1,601 positions: 26 tiles over 8 CTAs
    (4, 2, (165, 1), 9, 4),          # 11 tiles over 4; the other request has one tile, most of its CTAs none
    (8, 8, (150, 159, 160), 7, 4),   # hd 64; the last tile of the context nearly empty, full, and one position into the next
])
def test_split_attention_matches_the_oracle(heads, kv_heads, lens, beam, split, tmp_path):
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=2, n_q_heads=heads, n_kv_heads=kv_heads, n_items=50_000,
                     batch=len(lens), beam=beam, n_hist=max(lens), seed=21)
    case = Case(w)
    case.eng.prefill(case.hist_dev, torch.tensor(lens, dtype=torch.int32, device="cuda"))
    h = case.eng.get_hidden().cpu().numpy()
    out, launches = _attention_launches(lambda: case.eng.decode(beam, mode=1, trace=True), tmp_path / "trace.json")
    assert launches is None or launches and all(", 1, 2, true, true>" in name and grid[0] == split * kv_heads for name, grid in launches), launches
    ar = case.eng.decode(beam, mode=2)
    assert torch.equal(out["codes"], ar["codes"]) and torch.equal(out["count"], ar["count"])
    check_walk_against_trace(out, w.batch, w.L)
    beams, scores = out["trace"]["beams"].cpu().numpy(), out["trace"]["beam_scores"].cpu().numpy()
    for b, n in enumerate(lens):
        req = case.req(b, n)
        case._reqs[(b, None)] = req                      # (the ragged request is the one check_levels asks for)
        assert np.abs(h[b] - np.asarray(req.h, dtype=np.float64)).max() < hidden_tolerance(w)
        check_levels(case, b, beams[:, b], scores[:, b], beam, tol=tolerance(w))
    case.eng.close()
