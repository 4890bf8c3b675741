"""The same call on the same prefilled requests returns the same bits, whatever calls came before it."""
import pytest
import torch

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


# The token counts that earlier calls leave behind shape the tiling of later ones; the attention's kernels sum in different orders.
@pytest.mark.parametrize("hd,heads,kv_heads,batch,beam,n_hist", [(64, 28, 4, 5, 20, 50),     # 100 to 300 rows a pass
                                                                 (64, 8, 8, 64, 10, 50),     # 10 to 30 rows a request and KV head
                                                                 (64, 8, 2, 64, 10, 50),     # 40 to 120
                                                                 (128, 8, 2, 32, 20, 50),    # 80 to 240, one or two row tiles
                                                                 (64, 12, 4, 3, 11, 200)])   # long contexts, few requests
def test_repeated_calls_return_the_same_bits(hd, heads, kv_heads, batch, beam, n_hist):
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=2, d_model=hd * heads, n_q_heads=heads, n_kv_heads=kv_heads, n_items=50_000,
                     batch=batch, beam=beam, n_hist=n_hist)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):                          # (the engine reads the weights and histories on its stream)
        case = Case(w, stream=st).prefill()
    first, outs = {}, {m: case.eng.alloc_outputs(w.batch, w.beam, trace=True) for m in (binding.MODE_AR, binding.MODE_VERIFIED)}
    for mode in (binding.MODE_AR, binding.MODE_AR, binding.MODE_AR, binding.MODE_VERIFIED, binding.MODE_AR, binding.MODE_VERIFIED,
                 binding.MODE_VERIFIED, binding.MODE_VERIFIED):
        out = case.eng.decode(w.beam, mode=mode, out=outs[mode])
        torch.cuda.synchronize()
        got = [t.clone() for t in (out["codes"], out["scores"], out["count"], out["trace"]["beams"], out["trace"]["beam_scores"])]
        for a, b in zip(first.setdefault(mode, got), got):
            assert torch.equal(a, b), mode
    case.eng.close()
