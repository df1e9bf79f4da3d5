"""Bias gradients from partial column sums: the sum on its own, and the feed-forward layer's whose width is off 32."""
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests import gram_helpers as gh
from tests.test_gpu_gemm import ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [0, 4, 2, 1])
@pytest.mark.parametrize("rows,N", [(1, 8), (7, 40), (63, 1096), (64, 32), (65, 200), (513, 2304), (800, 3072), (5000, 100)])
def test_column_sums(rows, N, blocks):
    g = ctx()
    g.selftest_cluster_blocks(blocks)
    gen = torch.Generator(device="cuda").manual_seed(rows + N)
    part = torch.rand(rows, N, generator=gen, device="cuda") + 0.5
    out = torch.full((N,), 3.0, device="cuda")
    g.selftest_column_sums(part, out)
    g.sync()
    g.close()
    want = part.double().sum(0) + 3.0
    # n fp32 additions in any order: off by at most n * 2^-24 of the sum of the magnitudes
    assert ((out.double() - want).abs() <= (rows + 1) * 2.0 ** -24 * want).all()


def test_column_sums_do_not_depend_on_the_clusters_and_keep_their_chains_short():
    """64 rows far larger than the rest: an addition to them loses what a chain that does not hold them keeps."""
    rows, N = 32_768, 72
    part = torch.ones(rows, N, device="cuda")
    part[:64] = 2.0 ** 24
    part += torch.rand(rows, N, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    want, got = part.double().sum(0), []
    for blocks in (0, 8, 4, 2, 1):
        g = ctx()
        g.selftest_cluster_blocks(blocks)
        got.append(torch.zeros(N, device="cuda"))
        g.selftest_column_sums(part, got[-1])
        g.sync()
        g.close()
        assert torch.equal(got[-1], got[0])
    # an element passes rows / 512 additions of its chain, 3 of the chains, 7 of the warps, 7 of the parts and the last one, each
    # off by at most 2^-24 of a sum that is no larger than the whole
    assert ((got[0].double() - want).abs() <= (rows / 512 + 18) * 2.0 ** -24 * want).all()


@pytest.mark.parametrize("B,L", [(13, 20), (9, 60)])
def test_feed_forward_bias_of_a_width_off_32(B, L):
    """1096 columns: the last cluster of the sum has columns that do not exist, and the product before it ends in half-width units."""
    shape = synth.GramShape(name="b", dtype="bf16", n_items=1, l_t=1, vocab=1, d=128, n_heads=2, d_ff=8, n_layers=0, task="kt",
                            task_layers=1, task_heads=2, task_d_ff=1096, task_attn_only=False, B=B, L=L)
    tk = synth.task_params(shape, 3, sigma=0.1, plain=False)
    lab = synth.labels(5, B, L, 0.6)
    E = torch.randn(B, L, 128, generator=torch.Generator().manual_seed(B))
    th, e = orc.as_torch(tk), E.double().requires_grad_(True)
    orc.task_loss(th, e, lab, shape).backward()
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(tk))
    dE, loss = torch.empty(B * L, 128, device="cuda"), torch.empty(1, device="cuda")
    g.task(E.cuda().contiguous(), torch.from_numpy(lab).cuda(), B, dE, loss)
    g.sync()
    got = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    g.close()
    for name in ("t0.b1", "t0.bqkv", "t0.w1"):
        assert gh.rel_err(got[name], th[name].grad.numpy()) <= 2e-2, name          # bf16 operands, as in the whole steps' tests
