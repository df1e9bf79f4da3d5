"""The task module's input and head kernels at widths that allow 16-byte accesses and at widths that do not, and at batches
that leave some of a block's warps without a history."""
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads", [(6, 1), (10, 1), (12, 1), (132, 3), (260, 5)])
@pytest.mark.parametrize("B,L", [(1, 1), (3, 5), (37, 7)])
def test_task_gradients(d, heads, B, L):
    shape = synth.GramShape(name="t", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=heads, d_ff=4, n_layers=0, task="kt",
                            task_layers=1, task_heads=heads, task_d_ff=4, task_attn_only=True, B=B, L=L)
    tk = synth.task_params(shape, 3, sigma=0.1, plain=False)
    lab = synth.labels(5, B, L, 0.6)
    E = torch.randn(B, L, d, generator=torch.Generator().manual_seed(d + B))
    th, e = orc.as_torch(tk), E.double().requires_grad_(True)
    want = orc.task_loss(th, e, lab, shape)
    want.backward()
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(tk))
    dE, loss = torch.empty(B * L, d, device="cuda"), torch.empty(1, device="cuda")
    g.task(E.cuda().contiguous(), torch.from_numpy(lab).cuda(), B, dE, loss)
    g.sync()
    got = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    g.close()
    # fp32 sums of at most 259 x 260 terms: 2e-6 is what such models show, an order of magnitude above it
    assert abs(loss.item() - want.item()) <= 2e-5 * abs(want.item())
    assert gh.rel_err(dE.cpu().numpy(), e.grad.reshape(B * L, d).numpy()) <= 2e-5
    for name, t in th.items():
        w = t.grad.numpy()
        if abs(w).max() > 1e-9:                              # a one-row history has no gradient through its attention weights
            assert gh.rel_err(got[name], w) <= 2e-5, name
