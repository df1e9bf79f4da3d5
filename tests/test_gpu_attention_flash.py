"""Encoder and task attention at the lengths where the kernel changes: edges of 16-row tiles, of chunks, of the two launch
forms, texts of one and of many lengths, causal histories."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu

BASE = dict(dtype="bf16", vocab=50, d=128, n_heads=2, d_ff=128, n_layers=1, pooling="mean", task="kt", task_layers=1, task_heads=2,
            task_d_ff=128, task_attn_only=False, zipf_s=0.8)


def check_encoder(shape, lengths=None):
    """One layer's encodings and its VJP with random cotangents.  bf16 operands: 2e-2 on the worst parameter tensor, the
    bound of the whole-step tests (random cotangents, because a batch whose gradients nearly cancel says little)."""
    ce, tk, toks, _, _ = gh.make_inputs(shape, seed=6)
    g = gh.make_ctx(shape, ce, tk, toks)
    texts = toks
    if lengths is not None:
        g.set_item_lengths(lengths)
        texts = synth.ragged(toks, lengths)
    n = shape.n_items
    G = np.random.default_rng(1).standard_normal((n, shape.d)).astype(np.float32)
    th = orc.as_torch(ce)
    want = torch.stack([orc.ce_forward(th, texts[i], shape) for i in range(n)])
    want.backward(torch.from_numpy(G).double())
    items = torch.arange(n, dtype=torch.int32, device="cuda")
    H = torch.empty(n, shape.d, device="cuda")
    g.encode_unique(None, items, n, H, save_activations=True)
    g.zero_grads(binding.GRAM_MODULE_CE)
    g.encoder_backward(torch.from_numpy(G).cuda(), items, n)
    g.sync()
    got, _ = gh.gpu_grads(g, shape)
    g.close()
    assert gh.rel_err(H.cpu().numpy(), want.detach().numpy()) <= 2e-2
    err, name = gh.worst_rel_err(got, {k: t.grad.numpy() for k, t in th.items()})
    assert err <= 2e-2, name


@pytest.mark.parametrize("l_t", [65, 81, 96, 129, 144, 147, 160, 161, 177, 192, 193, 256])
def test_texts(l_t):
    check_encoder(synth.GramShape(name="t", n_items=9, l_t=l_t, B=9, L=1, **BASE))


@pytest.mark.parametrize("l_t", [150, 190, 240])
def test_texts_of_many_lengths(l_t):
    shape = synth.GramShape(name="v", n_items=24, l_t=l_t, B=24, L=1, **BASE)
    check_encoder(shape, synth.item_lengths(2, shape.n_items, l_t, 1))


@pytest.mark.parametrize("L", [65, 79, 96, 129, 145, 160, 175, 192, 200, 256])
def test_histories(L):
    shape = synth.GramShape(name="h", n_items=20, l_t=6, B=2, L=L, **BASE)
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=6)
    want = orc.gram_single_step(shape, ce, tk, toks, ids, lab)
    rep, gce, gtk = gh.gpu_single_step(shape, ce, tk, toks, ids, lab)
    assert abs(rep.loss - want["loss"]) <= 2e-2 * abs(want["loss"])
    for got, w in ((gce, want["grad_ce"]), (gtk, want["grad_task"])):
        err, name = gh.worst_rel_err(got, w)
        assert err <= 2e-2, name


@pytest.mark.parametrize("l_t", [66, 80, 96])
def test_texts_in_six_warps(l_t):
    """Heads of width 32 and 65 to 96 rows: blocks of six warps, one 16-row tile each."""
    check_encoder(synth.GramShape(name="s", n_items=9, l_t=l_t, B=9, L=1, **dict(BASE, n_heads=4)))
    check_encoder(synth.GramShape(name="s", n_items=9, l_t=l_t, B=9, L=1, **dict(BASE, n_heads=4)), synth.item_lengths(2, 9, l_t, 1))
