"""The mean over the predictions that are not padding, and the gradients that it divides, where every block of the task head counts them
for itself and where a launch of its own does (4096 positions and one more), a row a warp and several (1184 positions and one more, 9472
and some more), for rows that allow 16-byte accesses and rows that do not."""
import pytest
import torch

from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [32, 18])
@pytest.mark.parametrize("B,L", [(1, 1), (5, 51), (16, 74), (15, 79), (32, 128), (241, 17), (102, 93)])
def test_mean_over_real_predictions(B, L, d):
    shape = synth.GramShape(name="h", dtype="f32", n_items=1, l_t=1, vocab=1, d=d, n_heads=1, d_ff=4, n_layers=0, task="kt", task_layers=0,
                            task_heads=1, task_d_ff=4, task_attn_only=False, B=B, L=L)
    g = binding.Gram(binding.config_from_shape(shape))
    params = synth.task_params(shape, 3, sigma=0.1, plain=False)
    g.set_params(binding.GRAM_MODULE_TASK, synth.flatten(params))
    gen = torch.Generator().manual_seed(B * L)
    E = torch.randn(B, L, d, generator=gen)
    lab = torch.randint(0, 2, (B, L), generator=gen, dtype=torch.int32)
    n = torch.randint(1, L + 1, (B,), generator=gen)
    real = torch.arange(L)[None] < n[:, None]
    lab[~real] = -1
    dE, loss = torch.full((B * L, d), float("nan"), device="cuda"), torch.empty(1, device="cuda")
    g.task(E.cuda(), lab.cuda(), B, dE, loss)
    g.sync()
    grads = synth.unflatten(g.get_grads(binding.GRAM_MODULE_TASK), synth.task_param_spec(shape))
    g.close()
    p = {k: torch.from_numpy(v).double().requires_grad_() for k, v in params.items()}
    E64 = E.double().requires_grad_()
    prev = torch.cat([torch.full((B, 1), 2), lab[:, :-1].clamp(min=0).long()], 1)
    y = E64 + p["pos"].view(L, d) + p["resp"].view(3, d)[prev]
    z = y @ p["head_w"].view(d) + p["head_b"]
    want = torch.nn.functional.binary_cross_entropy_with_logits(z[real], lab[real].double())
    want.backward()
    # a mean of terms of about 0.7 in 32 bits: some hundred roundings of 2^-24 each
    assert abs(loss.item() - want.item()) <= 1e-5 * want.item()
    # A prediction's gradient (sigmoid - label) / count carries a quarter of its logit's error, (d + 4) roundings of 2^-24 of terms that
    # add up to some 6, and a few of the exponential and the division: below 4e-6 / count.  Sums over rows add a hundred roundings of
    # 2^-24 of the sizes added: together below 1e-5 of one per row.
    got = dE.cpu().double().view(B, L, d)
    w = p["head_w"].detach().view(d).abs()
    one = 1e-5 * w / int(real.sum())
    assert torch.equal(got[~real], torch.zeros_like(got[~real]))
    assert ((got - E64.grad).abs() <= one).all()
    rows_of = torch.stack([(real & (prev == k)).sum() for k in range(3)])
    bounds = {"pos": real.sum(0)[:, None] * one, "resp": rows_of[:, None] * one,
              "head_w": 1e-5 * y.detach()[real].abs().sum(0) / int(real.sum()), "head_b": torch.tensor(1e-5)}
    for name, bound in bounds.items():
        err = (torch.from_numpy(grads[name]).double().view(bound.shape) - p[name].grad.view(bound.shape)).abs()
        assert (err <= bound + 1e-12).all(), name
