"""Encoder and task attention at the lengths where the kernel changes: edges of 16-row tiles, of chunks, of the two launch
forms, texts of one and of many lengths, causal histories."""
import numpy as np
import pytest

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu

BASE = dict(dtype="bf16", vocab=50, d=128, n_heads=2, d_ff=128, n_layers=1, pooling="mean", task="kt", task_layers=1, task_heads=2,
            task_d_ff=128, task_attn_only=False, zipf_s=0.8)


def check(shape, lengths=None):
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=6)
    g = gh.make_ctx(shape, ce, tk, toks)
    texts = toks
    if lengths is not None:
        g.set_item_lengths(lengths)
        texts = synth.ragged(toks, lengths)
    want = orc.gram_single_step(shape, ce, tk, texts, ids, lab)
    import torch
    rep = g.step(torch.from_numpy(ids).cuda(), torch.from_numpy(lab).cuda(), shape.B)
    gce, gtk = gh.gpu_grads(g, shape)
    g.close()
    # bf16 operands: 2e-2 on the worst parameter tensor, the bound of the other whole-step tests
    assert abs(rep.loss - want["loss"]) <= 2e-2 * abs(want["loss"])
    for got, w in ((gce, want["grad_ce"]), (gtk, want["grad_task"])):
        err, name = gh.worst_rel_err(got, w)
        assert err <= 2e-2, name


@pytest.mark.parametrize("l_t", [65, 81, 96, 129, 144, 147, 160, 161, 177, 192, 193, 256])
def test_texts(l_t):
    # 80 predictions.  An element of the task module's weight gradients is a sum over the predictions whose addends carry up
    # to four roundings of 2^-9 each: its error is below 4 * 2^-9 * sum|a| / |sum a|, and with 18 addends of either sign the
    # ratio of the sums reached 2.6 on the largest element (2.06e-2); over 80 it stays below 2 where the element is largest.
    check(synth.GramShape(name="t", n_items=12, l_t=l_t, B=5, L=16, **BASE))


@pytest.mark.parametrize("l_t", [150, 190, 240])
def test_texts_of_many_lengths(l_t):
    shape = synth.GramShape(name="v", n_items=24, l_t=l_t, B=3, L=10, **BASE)
    check(shape, synth.item_lengths(2, shape.n_items, l_t, 1))


@pytest.mark.parametrize("L", [65, 79, 96, 129, 145, 160, 175, 192, 200, 256])
def test_histories(L):
    check(synth.GramShape(name="h", n_items=20, l_t=6, B=2, L=L, **BASE))
