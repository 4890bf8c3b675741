"""The prompt pass works on the real tokens of a batch of unequal histories, packed one request after another."""
import numpy as np
import pytest
import torch

from paper_2511_18793_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,batch,n_hist", [("fp32", 300, 20),      # several rounds of the offset sum, two chunks of requests
                                                ("bf16", 100, 50),      # two chunks, the tensor-core kernels
                                                ("bf16", 3, 300)])      # more than one tile of positions per request
def test_packed_prefill_equals_one_request_at_a_time(dtype, batch, n_hist):
    from gpu_helpers import Case, hidden_tolerance
    base = synth.WORKLOADS["tiny" if dtype == "fp32" else "small"]
    w = synth.scaled(base, n_layers=2, n_items=5_000, batch=batch, n_hist=n_hist)
    case = Case(w)
    rng = np.random.default_rng(3)
    lens = rng.integers(0, n_hist + 1, size=batch)
    lens[:3] = (n_hist, 0, 1)
    lens[-1] = n_hist
    n = torch.from_numpy(lens.astype(np.int32)).cuda()
    case.eng.prefill(case.hist_dev, n)
    together = case.eng.get_hidden().clone()
    for b in sorted({0, 1, 2, batch // 2, batch - 2, batch - 1}):
        case.eng.prefill(case.hist_dev[b:b + 1], n[b:b + 1])
        alone = case.eng.get_hidden()[0]
        if dtype == "fp32":      # the same sums in the same order whatever the other rows of a pass are: the same bits
            assert torch.equal(together[b], alone), b
        else:                    # the attention's kernel goes by the number of requests, and another order of its sums flips bf16
            # roundings downstream: two results, each within the bf16 rounding model's bound of the exact one
            assert (together[b] - alone).abs().max().item() < 2 * hidden_tolerance(w), b
    case.eng.close()
