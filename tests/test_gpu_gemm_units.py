"""The paired matrix product's GELU epilogue without the derivative."""
import numpy as np
import pytest
import torch

from tests import test_gpu_gemm as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(512, 768, 768), (1000, 768, 136), (520, 1032, 128), (136, 200, 72), (19_000, 768, 72)])
def test_gelu_without_its_derivative(M, N, K):
    g = base.ctx()
    gen = torch.Generator(device="cpu").manual_seed(M + N + K)
    A = (torch.randn(M, K, generator=gen) * 0.5).to(torch.bfloat16).to(base.DEV)
    B = (torch.randn(N, K, generator=gen) * (2.0 / np.sqrt(K))).to(torch.bfloat16).to(base.DEV)
    bias = (torch.randn(N, generator=gen) * 0.3).to(base.DEV)
    C = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=base.DEV)
    g.gemm_bf16_epilogue(A, 1, B, 1, C, M, N, K, bias=bias, gelu=True)
    g.sync()
    g.close()
    want, _ = base._erf_gelu((A.double() @ B.double().T + bias.double()).cpu())
    scale = want.abs().max().item()
    # the bound of the epilogue with the derivative: sums of K products, the rational erf, the result's rounding
    assert (C.double().cpu() - want).abs().max().item() <= 1e-4 * np.sqrt(K) + 2.0 ** -8 * scale + 2e-6 * scale + 4e-7 * scale + 2e-6
