"""Kernels whose warps read rows through a ring of bulk copies, when a wait for a row runs out (the kernel decides so itself after
a number of rows; the copies do arrive): the error is reported, nothing of the sums is left behind, the context stays usable."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests.test_gpu_index import index_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rows", [0, 1])
def test_layernorm_backward_gives_up(dtype, rows):
    """3000 rows: more than one for each of the 8 x 148 warps, so that with rows = 1 every block has sums when it gives up."""
    B, L, d = 60, 50, 128
    shape = synth.GramShape(name="r", dtype=dtype, n_items=1, l_t=1, vocab=1, d=d, n_heads=2, d_ff=64, n_layers=0, task="kt", task_layers=1,
                            task_heads=2, task_d_ff=64, task_attn_only=False, B=B, L=L)
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(synth.task_params(shape, 3, sigma=0.1, plain=False)))
    E = torch.randn(B, L, d, generator=torch.Generator().manual_seed(1)).cuda()
    lab = torch.from_numpy(synth.labels(5, B, L, 0.6)).cuda()
    dE, loss = torch.empty(B * L, d, device="cuda"), torch.empty(1, device="cuda")

    def grads():
        g.task(E, lab, B, dE, loss)
        g.sync()
        return synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))

    want = grads()
    assert np.abs(want["t0.ln2_g"]).max() > 0
    g.selftest_ring_rows(rows)
    g.task(E, lab, B, dE, loss)
    with pytest.raises(binding.GramError, match="GRAM_ERR_TIMEOUT"):
        g.sync()
    got = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    for name in ("t0.ln2_g", "t0.ln2_b", "t0.ln1_g", "t0.ln1_b"):
        assert not got[name].any(), name
    g.selftest_ring_rows(-1)
    again = grads()
    for name, w in want.items():
        assert np.array_equal(again[name], w), name
    g.close()


@pytest.mark.parametrize("rows", [0, 7])
def test_segment_sums_give_up(rows):
    """A call over few items after one over many: what the first left in the workspace (its items that run over the end of a
    chunk) names rows that the second does not have.  The rows after its own are the test's, and stay as they are."""
    P, d, many = 40_000, 768, 5000
    g = index_ctx(P, many, d)
    dE = torch.rand(P, d, generator=torch.Generator().manual_seed(2)).cuda()

    def index(n):
        ids = np.sort(np.arange(P, dtype=np.int32) % n)
        unique, _, perm, seg = orc.unique_inverse(ids)
        return len(unique), torch.from_numpy(perm.astype(np.int32)).cuda(), torch.from_numpy(seg.astype(np.int32)).cuda()

    G = torch.zeros(many, d, device="cuda")
    U, perm, seg = index(many)
    g.accumulate(dE, perm, seg, U, G)
    g.sync()
    U, perm, seg = index(3)
    G.fill_(-7.0)
    g.selftest_ring_rows(rows)
    g.accumulate(dE, perm, seg, U, G)
    with pytest.raises(binding.GramError, match="GRAM_ERR_TIMEOUT"):
        g.sync()
    assert (G[U:] == -7.0).all()
    g.selftest_ring_rows(-1)
    g.accumulate(dE, perm, seg, U, G)
    g.sync()
    want = torch.stack([dE[perm[seg[u]:seg[u + 1]].long()].double().sum(0) for u in range(U)])
    assert ((G[:U] - want).abs() <= 1e-5 * want.abs()).all()        # sums of 13 000 positive terms over chunks of 17
    g.close()
