"""Texts of three and more attention tiles, with more (sequence, tile, head) items than thread blocks."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as O
from paper_2204_04179_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l_t,shortest,n", [(271, 271, 90), (257, 1, 120), (400, 120, 70), (512, 512, 40)])
def test_many_long_texts(l_t, shortest, n):
    """A block then takes several items of at least three key tiles one after the other.  bf16 operands: the encodings
    of one layer are within 1 % of the 64-bit ones (2^-9 per rounding, a handful of roundings on the way)."""
    shape = synth.GramShape(name="long", dtype="bf16", n_items=n, l_t=l_t, vocab=200, d=128, n_heads=2, d_ff=128, n_layers=1,
                            pooling="mean", task="kt", task_heads=2, B=n, L=1)
    par = synth.encoder_params(shape, 3, sigma=0.1, plain=False)
    tokens = synth.item_tokens(3, n, l_t, shape.vocab)
    lengths = synth.item_lengths(3, n, l_t, shortest)
    g = binding.Gram(binding.config_from_shape(shape))
    try:
        g.set_params(binding.GRAM_MODULE_CE, synth.flatten(par))
        g.set_item_tokens(tokens)
        if shortest < l_t:
            g.set_item_lengths(lengths)
        items = torch.arange(n, dtype=torch.int32, device="cuda")
        H = torch.zeros(n, shape.d, device="cuda")
        g.encode_unique(None, items, n, H)
        g.sync()
        texts = synth.ragged(tokens, lengths) if shortest < l_t else list(tokens)
        want = O.encode_all(shape, par, texts, range(n))
        assert np.linalg.norm(H.cpu().numpy() - want) <= 1e-2 * np.linalg.norm(want)
    finally:
        g.close()
