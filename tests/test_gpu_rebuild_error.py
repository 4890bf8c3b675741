"""A rebuild of the catalogue's tables that CUDA refuses: an engine on the legacy default stream, while a stream that
synchronises with that one is being captured (every launch returns an error code; nothing runs)."""
import numpy as np
import pytest
import torch

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


def _refused_rebuild(eng):
    from cuda.bindings import runtime as rt
    torch.cuda.synchronize()
    err, st = rt.cudaStreamCreate()
    assert err == rt.cudaError_t.cudaSuccess
    (err,) = rt.cudaStreamBeginCapture(st, rt.cudaStreamCaptureMode.cudaStreamCaptureModeGlobal)
    assert err == rt.cudaError_t.cudaSuccess
    try:
        with pytest.raises(binding.NezhaError) as e:
            eng.build_hashset()
    finally:
        rt.cudaStreamEndCapture(st)
        rt.cudaStreamDestroy(st)
    return e.value


@pytest.mark.parametrize("n", [5_000, 1_600_000])              # one pass, and by parts
def test_the_next_calls_are_not_refused_too(n):
    T = (128, 128, 64, 16)
    rng = np.random.default_rng(n)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["tiny"], L=4, T=T, n_items=n, batch=1, beam=2, n_hist=1)
    case = Case(w, catalog=cat, hist=cat[:1, None])
    _refused_rebuild(case.eng)
    keys = case.eng.pack(case.cat_dev)
    assert case.eng.build_hashset() == case.n_unique
    assert case.eng.probe(keys).all().item()
    case.eng.close()


@pytest.mark.parametrize("n", [5_000, 1_600_000])
def test_no_call_reads_tables_whose_rebuild_failed(n):
    T = (128, 128, 64, 16)
    rng = np.random.default_rng(n)
    cat = np.stack([rng.integers(0, t, size=n) for t in T], axis=1).astype(np.int32)
    w = synth.scaled(synth.WORKLOADS["tiny"], L=4, T=T, n_items=n, batch=1, beam=2, n_hist=1)
    case = Case(w, catalog=cat, hist=cat[:1, None]).prefill()
    keys = case.eng.pack(case.cat_dev)
    _refused_rebuild(case.eng)
    for call in (lambda: case.eng.probe(keys), lambda: case.eng.decode(2), lambda: case.prefill()):
        with pytest.raises(binding.NezhaError) as e:
            call()
        assert binding.STATUS_NAMES[e.value.status] == "ERR_STATE"
    case.eng.build_hashset()
    assert case.eng.probe(keys).all().item()
    case.prefill()
    case.eng.decode(2)
    case.eng.close()
