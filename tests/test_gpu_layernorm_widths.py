"""LayerNorm backward at the widths of its row rings (a float4 per lane and slot: 128 columns each), full and with idle lanes, over more
rows than a ring holds; and the task's row kernels on encodings that do not start on 16 bytes."""
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu


def check(d, heads, B, L, shift=0):
    shape = synth.GramShape(name="t", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=heads, d_ff=4, n_layers=0, task="kt",
                            task_layers=1, task_heads=heads, task_d_ff=8, task_attn_only=False, B=B, L=L)
    tk = synth.task_params(shape, 3, sigma=0.1, plain=False)
    lab = synth.labels(5, B, L, 0.6)
    E = torch.randn(B, L, d, generator=torch.Generator().manual_seed(d + B))
    th, e = orc.as_torch(tk), E.double().requires_grad_(True)
    want = orc.task_loss(th, e, lab, shape)
    want.backward()
    g = binding.Gram(binding.config_from_shape(shape))
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(tk))
    x, dE = (torch.empty(B * L * d + shift, device="cuda")[shift:] for _ in range(2))
    x.copy_(E.reshape(-1))
    loss = torch.empty(1, device="cuda")
    g.task(x, torch.from_numpy(lab).cuda(), B, dE, loss)
    g.sync()
    got = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    g.close()
    # fp32 sums of up to 4500 rows or 1024 columns: a few 1e-6 is what such models show, an order of magnitude above it
    assert abs(loss.item() - want.item()) <= 2e-5 * abs(want.item())
    assert gh.rel_err(dE.cpu().numpy().reshape(-1, d), e.grad.reshape(-1, d).numpy()) <= 2e-5
    err, name = gh.worst_rel_err(got, {k: t.grad.numpy() for k, t in th.items()})
    assert err <= 2e-5, name


@pytest.mark.parametrize("d,heads", [(128, 2), (132, 3), (256, 4), (512, 8), (516, 12), (768, 12), (900, 15), (1020, 17), (1024, 16)])
def test_widths(d, heads):
    check(d, heads, 90, 50)


@pytest.mark.parametrize("shift", [1, 2])
def test_rows_that_do_not_start_on_16_bytes(shift):
    check(64, 2, 5, 7, shift)
