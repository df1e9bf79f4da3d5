"""Embedding, LayerNorm and mean pooling of fp32 encoders: rows of few and of many float4s, one row and more rows than are fetched
ahead, texts of one and of many lengths, the caller's encodings and cotangents on and off 16 bytes."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,l_t,pooling,ragged,shift", [(36, 3, 1, "mean", False, 1), (36, 3, 7, "mean", True, 0), (132, 3, 33, "mean", True, 2),
                                                             (256, 4, 70, "mean", False, 0), (1024, 16, 9, "mean", True, 3),
                                                             (128, 2, 5, "cls", True, 1), (128, 2, 1, "cls", False, 3)])
def test_encodings_and_their_gradients(d, heads, l_t, pooling, ragged, shift):
    shape = synth.GramShape(name="p", dtype="f32", n_items=11, l_t=l_t, vocab=50, d=d, n_heads=heads, d_ff=2 * d, n_layers=1,
                            pooling=pooling, task="kt", task_layers=0, task_heads=1, task_d_ff=4, B=11, L=1)
    ce, tk, toks, _, _ = gh.make_inputs(shape, seed=8)
    g = gh.make_ctx(shape, ce, tk, toks)
    texts, n = toks, shape.n_items
    if ragged:
        lengths = synth.item_lengths(4, n, l_t, 1)
        g.set_item_lengths(lengths)
        texts = synth.ragged(toks, lengths)
    G = np.random.default_rng(2).standard_normal((n, d)).astype(np.float32)
    th = orc.as_torch(ce)
    want = torch.stack([orc.ce_forward(th, texts[i], shape) for i in range(n)])
    want.backward(torch.from_numpy(G).double())
    items = torch.arange(n, dtype=torch.int32, device="cuda")
    H, Gd = (torch.zeros(n * d + shift, device="cuda")[shift:] for _ in range(2))
    Gd.copy_(torch.from_numpy(G).reshape(-1))
    bare = torch.zeros(n, d, device="cuda")
    g.encode_unique(None, items, n, bare)                          # nothing kept for a backward pass: the same encodings
    g.encode_unique(None, items, n, H, save_activations=True)
    g.zero_grads(binding.GRAM_MODULE_CE)
    g.encoder_backward(Gd, items, n)
    g.sync()
    got, _ = gh.gpu_grads(g, shape)
    g.close()
    assert torch.equal(H.view(n, d), bare)
    # fp32 sums over at most 1024 columns or 770 rows: an order of magnitude above what such models show
    assert gh.rel_err(H.cpu().numpy().reshape(n, d), want.detach().numpy()) <= 2e-5
    err, name = gh.worst_rel_err(got, {k: t.grad.numpy() for k, t in th.items()})
    assert err <= 2e-5, name
