"""Weight gradients of fp32 contexts by themselves against 64 bits: as exact as the chains of additions that a product on its own takes.

One attention-only task layer over histories of one position.  The query, key and value weights are zero and the head reads a column
that is zero in every row, so that every prediction is 1/2 and the gradient that reaches the value rows is one rounded product per
element: what is left of the error is the sum over the rows."""
import numpy as np
import pytest
import torch

from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


# width, rows, and how a product alone adds up dWqkv: the longest chain of additions, the groups of a block and the parts of a cluster
# that come after it
@pytest.mark.parametrize("d,rows,chain,groups,parts", [(64, 912, 32, 4, 8), (64, 4096, 64, 4, 16), (64, 6400, 128, 4, 16), (96, 3848, 256, 1, 16),
                                                       (96, 2952, 192, 1, 16), (128, 3000, 384, 1, 8), (32, 9000, 160, 4, 16), (64, 30, 30, 1, 1)])
def test_value_weight_gradient(d, rows, chain, groups, parts):
    shape = synth.GramShape(name="w", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=1, d_ff=4, n_layers=0, task="kt", task_layers=1,
                            task_heads=2, task_d_ff=4, task_attn_only=True, B=rows, L=1)
    params = {k: np.zeros_like(v) for k, v in synth.task_params(shape, 3).items()}
    rng = np.random.default_rng(d + rows)
    w_out = rng.standard_normal(d).astype(np.float32)
    params["head_w"].reshape(-1)[0] = 1.0
    params["t0.wo"].reshape(d, d)[0] = w_out
    x = rng.standard_normal((rows, d)).astype(np.float32)
    x[:, 0] = 0.0
    lab = rng.integers(0, 2, (rows, 1)).astype(np.int32)
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(params))
    dE, loss = torch.empty(rows, d, device="cuda"), torch.empty(1, device="cuda")
    g.task(torch.from_numpy(x).cuda(), torch.from_numpy(lab).cuda(), rows, dE, loss)
    g.sync()
    grads = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    g.close()
    share = (np.float32(0.5) - lab.astype(np.float32)) * (np.float32(1.0) / np.float32(rows))
    dv = (share * w_out[None]).astype(np.float64)                    # one rounding each, as in the product with one term that is not zero
    want = dv.T @ x.astype(np.float64)
    got = np.asarray(grads["t0.wqkv"], np.float64).reshape(3 * d, d)[2 * d:]
    # A sum of n terms of either sign, rounded at every step: 0.425 x 2^-24 of the partial sum's size each (a mantissa uniform over its
    # logarithm), over the chain, the groups and the parts; a quarter on top for the columns at hand, and the smallest result of 24 bits.
    bound = 1.25 * 0.425 * 2.0 ** -24 * ((chain + groups + parts) / 2) ** 0.5 + 2.0 ** -26
    assert np.linalg.norm(got - want) <= bound * np.linalg.norm(want)
