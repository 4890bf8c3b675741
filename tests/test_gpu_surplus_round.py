"""A round that was queued for nothing costs its launches, not a pass over the weights."""
import statistics

import pytest
import torch

from paper_2511_18793_b200 import binding, synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


def test_a_surplus_round_does_not_stream_the_weights():
    w = synth.scaled(synth.WORKLOADS["paper"], n_layers=8, n_items=50_000, batch=1)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):                          # (the engine reads the weights and histories on its stream)
        case = Case(w, stream=st).prefill()
        beams = case.eng.decode(w.beam, mode=binding.MODE_AR, trace=True)["trace"]["beams"].clone()
        tree = beams, (beams[:, :, :, 0] >= 0).sum(dim=2).to(torch.int32).contiguous()
    out = case.eng.alloc_outputs(1, w.beam)
    torch.cuda.synchronize()

    def plain():
        return case.eng.decode(w.beam, mode=binding.MODE_AR, out=out)["stats"].rounds

    def drafted():
        return case.eng.decode(w.beam, mode=binding.MODE_VERIFIED, out=out)["stats"].rounds

    def accepted():
        return case.eng.decode_with_draft_tree(w.beam, *tree, out=out)["stats"].rounds

    def time(*calls):
        """Median us of the last of the calls, the others made in front of it."""
        us = []
        for _ in range(15):
            for c in calls[:-1]:
                assert c() == 2
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(st)
            rounds = calls[-1]()
            b.record(st)
            b.synchronize()
            us.append(a.elapsed_time(b) * 1e3)
        assert rounds == (2 if calls[-1] is plain else 1)
        return statistics.median(us[4:])

    one, two = time(accepted), time(plain)
    surplus = time(drafted, accepted) - one              # (the call queues as many rounds as the one before it needed)
    print(f"one round {one:.0f} us, two {two:.0f}, a surplus one {surplus:.0f}")
    assert surplus < 0.6 * two / 2                       # (0.84 of a round with the weights read, 0.38 without)
    case.eng.close()
