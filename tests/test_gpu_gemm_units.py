"""Work units of the paired matrix product: whole waves followed by a last one of half-width units, K ranges of several accumulator
chains, the GELU epilogue without the derivative."""
import numpy as np
import pytest
import torch

from paper_2204_04179_b200 import binding
from tests import test_gpu_gemm as base

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["gelu", "dgelu", "res", "res_ln", "res_ln_copy", "bias_f32", "plain_bf16"])
@pytest.mark.parametrize("M,N,K", [(19_000, 768, 72), (6400, 1096, 136), (3000, 1800, 1032)])
def test_last_wave_of_halves(M, N, K, kind):
    """225, 125 and 96 tiles over 74 pairs of SMs: whole units, then halves of 3, 51 (too many: whole) and 22 tiles, ragged at the
    lower and right edges (a half that lies outside the matrix among them)."""
    base.test_gemm_epilogues_against_float64(M, N, K, kind)


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


@pytest.mark.parametrize("M,N,K", [(768, 768, 9000), (3072, 768, 4104), (1536, 768, 2056), (2048, 2048, 136), (2304, 2304, 1104), (264, 520, 3000),
                                   (264, 1096, 9000), (1000, 1800, 5000), (4872, 1096, 12_400)])
def test_chains_of_a_weight_gradient(M, N, K):
    """C += A^T B over K rows: several chains per unit and parts, one part alone, fewer k-blocks than chains would take; narrow columns
    (520: no pairs of SMs, no chains); ragged rows and columns with several chains, in parts and, over 100 tiles, with half-width units."""
    g = base.ctx()
    gen = torch.Generator(device=base.DEV).manual_seed(M + N + K)
    A = (torch.randn(K, M, generator=gen, device=base.DEV) * 0.5).to(torch.bfloat16)
    B = (torch.randn(K, N, generator=gen, device=base.DEV) * 0.5).to(torch.bfloat16)
    C = torch.full((M, N), 2.0, device=base.DEV)
    g.gemm_bf16(A, 0, B, 0, C, None, 1, M, N, K)
    g.sync()
    g.close()
    want = A.double().T @ B.double() + 2.0
    # as in the products' own test: sums of K products of bf16 values
    assert (C.double() - want).abs().max().item() <= 1e-4 * np.sqrt(K)


def test_parts_where_one_tile_leaves_the_chip_empty():
    """256 x 256 over 16 k-blocks: two chains.  One after the other would halve the few units there are, so they stay two parts:
    the product and the sum of its parts, two launches."""
    g = base.ctx()
    A, B = (torch.ones(1024, 256, dtype=torch.bfloat16, device=base.DEV) for _ in range(2))
    C = torch.zeros(256, 256, device=base.DEV)
    before = g.launch_count()
    g.gemm_bf16(A, 0, B, 0, C, None, 1, 256, 256, 1024)
    g.sync()
    assert g.launch_count() - before == 2
    g.close()
    assert (C == 1024).all()


def _long_sum_error(M, N, K, d, d_ff):
    """Relative error of A^T B over K rows of values of mostly one sign, in a context of width d, which sizes the workspace."""
    cfg = binding.GramConfig()
    cfg.n_items = cfg.P_max = 8
    cfg.d, cfg.d_ff = d, d_ff
    g = binding.Gram(cfg)
    gen = torch.Generator(device=base.DEV).manual_seed(5)
    A = (torch.randn(K, M, generator=gen, device=base.DEV) + 1).to(torch.bfloat16)
    B = (torch.randn(K, N, generator=gen, device=base.DEV) + 1).to(torch.bfloat16)
    C = torch.zeros(M, N, device=base.DEV)
    g.gemm_bf16(A, 0, B, 0, C, None, 1, M, N, K)
    g.sync()
    g.close()
    want = torch.zeros(M, N, dtype=torch.float64, device=base.DEV)
    for o in range(0, K, 8192):
        want += A[o:o + 8192].double().T @ B[o:o + 8192].double()
    return ((C - want).norm() / want.norm()).item()


@pytest.mark.parametrize("M,N", [(4864, 1024), (4872, 1096)])
def test_chains_where_the_tiles_fill_the_chip(M, N):
    """76 and 100 tiles, no parts: 65 536 rows in six chains, each of which loses at most 2^-24 per 16-term step."""
    assert _long_sum_error(M, N, 65_536, 768, 3072) <= 65_536 / 16 / 6 * 2.0 ** -24


def test_chains_of_a_small_workspace():
    """As many chains as with a model's workspace, so the same losses; only the few sums of chains are put together otherwise."""
    small, model = _long_sum_error(3072, 768, 65_536, 8, 0), _long_sum_error(3072, 768, 65_536, 768, 3072)
    assert abs(small - model) <= 20 * 2.0 ** -24
