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


# A product of at most 48 rows: its row scales are one warp's work and another's operand, its parts come from other CTAs.
@pytest.mark.parametrize("n_hist", [1, 6, 10])           # 9, 29 and 45 rows a prompt pass
def test_passes_of_few_rows_return_the_same_bits_many_times(n_hist):
    w = synth.scaled(synth.WORKLOADS["paper"], n_layers=2, L=4, T=(64,) * 4, n_items=50_000, batch=1, beam=10, n_hist=n_hist)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        case = Case(w, stream=st)
    out = {m: case.eng.alloc_outputs(1, w.beam) for m in (binding.MODE_AR, binding.MODE_VERIFIED)}
    first = None
    for _ in range(150):
        case.prefill()
        got = [case.eng.get_hidden()]
        for mode, o in out.items():
            got += [case.eng.decode(w.beam, mode=mode, out=o)[k].clone() for k in ("codes", "scores")]
        torch.cuda.synchronize()
        first = first or [t.clone() for t in got]
        for a, b in zip(first, got):
            assert torch.equal(a, b)
    assert torch.isfinite(first[0]).all()
    case.eng.close()


# A warp gives a tile of K and V back to the copies of the next while its last loads of that tile may be under way.
@pytest.mark.parametrize("hd,kv_heads,batch,beam,n_hist,level,calls", [
    (64, 8, 64, 10, 50, 1, 12_000), (64, 8, 64, 10, 50, 2, 12_000),     # 16-row CTAs, two warps that take every second tile
    (128, 4, 64, 10, 50, 2, 6_000),
    (64, 2, 64, 12, 50, 1, 6_000), (64, 8, 64, 40, 50, 1, 6_000),       # 48 and 40 rows, every warp all tiles
    (64, 2, 2, 10, 400, 1, 6_000)])                                     # tiles split over a cluster
def test_a_pass_returns_the_same_bits_thousands_of_times(hd, kv_heads, batch, beam, n_hist, level, calls):
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, n_q_heads=512 // hd, n_kv_heads=kv_heads, n_items=50_000, batch=batch, beam=beam,
                     n_hist=n_hist)
    case = Case(w).prefill()
    g = torch.Generator(device="cuda").manual_seed(1)
    prefixes = torch.randint(0, 256, (batch, beam, level), dtype=torch.int32, device="cuda", generator=g)
    first = case.eng.primary_logits(beam, level, prefixes).clone()
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(calls):
        bad += (case.eng.primary_logits(beam, level, prefixes) != first).any()
    assert torch.isfinite(first).all() and int(bad) == 0
    case.eng.close()
