"""The CUDA-core GEMM at odd sizes, and its two forms against each other."""
import numpy as np
import pytest
import torch

from paper_2511_18793_b200 import synth
from gpu_helpers import Case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return Case(synth.scaled(synth.WORKLOADS["tiny"], n_layers=1, batch=1, n_hist=1))


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (17, 5, 7), (16, 16, 128), (40, 64, 130), (33, 31, 257), (20, 192, 64), (700, 50, 64)])
def test_fp32_gemm(ctx, M, N, K):
    g = torch.Generator(device="cuda"); g.manual_seed(M * 7 + N * 3 + K)
    big = torch.randn(64 * 97, K, generator=g, device="cuda")     # more than 96 tiles of 64 x 64: the large form
    W = torch.randn(N, K, generator=g, device="cuda")
    bias = torch.randn(N, generator=g, device="cuda")
    A = big[:M].contiguous()
    ref = A.double().cpu().numpy() @ W.double().cpu().numpy().T
    # K products of unit variance summed in order: an error of at most K * 2^-24 of the sum of their magnitudes
    bound = K * 2.0 ** -24 * (np.abs(A.double().cpu().numpy()) @ np.abs(W.double().cpu().numpy()).T) + 1e-6
    full = torch.empty(big.shape[0], N, device="cuda")
    ctx.eng.gemm(big, W, full, epilogue=1)
    out = torch.empty(M, N, device="cuda")
    for epilogue in (0, 1):
        ctx.eng.gemm(A, W, out.fill_(float("nan")), epilogue=epilogue)
        assert torch.equal(out, full[:M])                          # one order of summation, whatever the form
        assert (np.abs(out.double().cpu().numpy() - ref) <= bound).all()
    acc = full[:M].clone()
    ctx.eng.gemm(A, W, acc, epilogue=2)
    assert torch.equal(acc, out + out)
    ctx.eng.gemm(A, W, acc, epilogue=3, bias=bias)
    assert np.abs(acc.double().cpu().numpy() - np.tanh(ref + bias.double().cpu().numpy())).max() <= bound.max() + 1e-6
    ctx.eng.sync()
