"""What a traced decode call leaves in the trace's beam sets, and when."""
import pytest
import torch

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [binding.MODE_VERIFIED, binding.MODE_AR])
def test_trace_is_complete_when_the_call_returns(mode):
    """The call synchronises: nothing of it is left on the engine's stream, and another stream may read the trace at once."""
    w = synth.scaled(synth.WORKLOADS["tiny"], n_layers=1, L=8, T=(16,) * 8, batch=512, beam=128, n_hist=1)   # 17 MB of beam sets
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(st):              # (the engine reads the weights and histories on its stream)
        case = Case(w, stream=st).prefill()
    out = case.eng.alloc_outputs(w.batch, w.beam, trace=True)
    beams = out["trace"]["beams"]
    for _ in range(4):                       # eager, captured, replayed
        beams.fill_(-7)
        torch.cuda.synchronize()
        case.eng.decode(w.beam, mode=mode, out=out)
        assert st.query()
        with torch.cuda.stream(other):
            seen = beams.clone()
        torch.cuda.synchronize()
        assert torch.equal(seen, beams) and (beams >= -1).all().item()
    case.eng.close()


def test_draft_mode_leaves_the_true_beam_sets_alone():
    """Mode 0 has no true beam sets: an earlier call's are not handed out as its own."""
    w = synth.scaled(synth.WORKLOADS["small"], n_layers=1, n_items=20_000, batch=3, n_hist=5)
    case = Case(w).prefill()
    case.eng.decode(w.beam, mode=binding.MODE_VERIFIED)
    out = case.eng.alloc_outputs(w.batch, w.beam, trace=True)
    for t in out["trace"].values():
        t.fill_(-7)
    torch.cuda.synchronize()
    case.eng.decode(w.beam, mode=binding.MODE_DRAFT, out=out)
    for name, t in out["trace"].items():
        assert (t == (-7 if name in ("beams", "beam_scores") else -1)).all().item(), name
    case.eng.close()
