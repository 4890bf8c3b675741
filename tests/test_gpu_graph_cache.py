"""Which decode calls replay a captured graph, read off the CUDA runtime calls that they make."""
import collections

import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


def _runtime_calls(call):
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    calls = collections.Counter(e.name for e in p.events() if e.name.startswith("cuda"))
    if not calls:
        pytest.skip("no activity records: another profiler holds the process")
    return calls


def _replayed(calls):
    return calls["cudaGraphLaunch"] == 1 and calls["cudaGraphInstantiate"] == 0 and calls["cudaLaunchKernelExC"] == 0


def _engines(**kw):
    """The same engine twice: on a stream of its own, and on the default stream, which replays nothing."""
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=2, T=(16,) * 4, n_items=20_000, batch=2, beam=5, n_hist=100, **kw)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):              # (the engine reads the weights on its stream)
        case = Case(w, stream=st)
    torch.cuda.synchronize()
    return case, Case(w, weights=case.weights, catalog=case.catalog, hist=case.hist)


def test_histories_of_other_lengths_replay_the_same_graph():
    case, eager = _engines()
    out = case.eng.alloc_outputs(2, 5)
    torch.cuda.synchronize()
    for i, n in enumerate((100, 100, 100, 100, 99, 57, 100, 3)):
        hist, lens = case.hist_dev[:, :n].contiguous(), torch.full((2,), n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for c in (case, eager):
            c.eng.prefill(hist, lens)
        torch.cuda.synchronize()
        calls = _runtime_calls(lambda: case.eng.decode(5, mode=binding.MODE_AR, out=out))
        assert i < 3 or _replayed(calls), (n, calls)
        want = eager.eng.decode(5, mode=binding.MODE_AR)
        for k in ("codes", "scores", "count"):
            assert torch.equal(out[k], want[k]), (n, k)
        assert (out["count"] > 0).all().item()
    case.eng.close()
    eager.eng.close()


def test_the_graphs_that_are_kept_are_bounded():
    """A program that brings other result buffers to every call: the oldest graphs are given back."""
    case, eager = _engines()
    torch.cuda.synchronize()
    for c in (case, eager):
        c.prefill()
    counts = torch.zeros(300, 2, dtype=torch.int32, device="cuda")
    out = case.eng.alloc_outputs(2, 5)
    torch.cuda.synchronize()

    def decode(i):
        case.eng.decode(5, mode=binding.MODE_AR, out={**out, "count": counts[i]})

    for i in range(300):
        for _ in range(3 if i % 50 == 0 else 1):
            decode(i)
    want = eager.eng.decode(5, mode=binding.MODE_AR)
    assert torch.equal(out["codes"], want["codes"]) and torch.equal(out["scores"], want["scores"])
    assert torch.equal(counts, want["count"].expand(300, 2))
    assert _replayed(_runtime_calls(lambda: decode(250)))                  # captured 50 buffers ago
    assert not _replayed(_runtime_calls(lambda: decode(0)))                # 300 ago
    decode(0)
    assert _replayed(_runtime_calls(lambda: decode(0)))
    assert torch.equal(counts[0], want["count"])
    case.eng.close()
    eager.eng.close()


def test_calls_with_other_trace_buffers_are_told_apart():
    """Trace buffers whose addresses differ in ways that cancel out in beams ^ 2 tree_codes."""
    case, eager = _engines()
    torch.cuda.synchronize()
    case.prefill()
    R, L, S = 3, 4, 1 << 12                                                # a buffer is less than 4 KB
    block = torch.empty(16 * S, dtype=torch.uint8, device="cuda")
    base = -block.data_ptr() % (8 * S)
    out = case.eng.alloc_outputs(2, 5, trace=True)

    def at(offset, like):
        return block[base + offset:base + offset + like.numel() * 4].view(torch.int32).view(like.shape)

    for i in range(2):
        trace = {**out["trace"], "beams": at(2 * S * i, out["trace"]["beams"]), "tree_codes": at(4 * S + S * i, out["trace"]["tree_codes"])}
        for _ in range(4):
            trace["tree_codes"].fill_(-7)
            torch.cuda.synchronize()
            case.eng.decode(5, mode=binding.MODE_VERIFIED, out={**out, "trace": trace})
            assert (trace["tree_codes"] >= -1).all().item() and trace["tree_codes"].shape == (R, L, 2, 5, L)
    case.eng.close()
    eager.eng.close()
