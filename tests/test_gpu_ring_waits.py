"""Kernels whose warps read rows through a ring of bulk copies, when a wait for a row runs out (the kernel decides so itself after
a number of rows; the copies do arrive): the error is reported, nothing of the sums is left behind, the context stays usable."""
import numpy as np
import pytest
import torch

from paper_2204_04179_b200 import binding, synth

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
