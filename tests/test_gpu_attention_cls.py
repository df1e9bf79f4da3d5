"""Token-0 pooling with heads of width 64: the last layer's attention runs with one query row per item."""
import pytest

from paper_2204_04179_b200 import synth
from tests.test_gpu_attention_flash import BASE, check_encoder

pytestmark = pytest.mark.gpu


def shape(l_t, n_layers, n_items=21):
    return synth.GramShape(**dict(BASE, name="c", n_items=n_items, l_t=l_t, n_layers=n_layers, pooling="cls", B=n_items, L=1))


@pytest.mark.parametrize("n_layers", [1, 2])
@pytest.mark.parametrize("l_t", [2, 3, 15, 17, 64, 65, 130])
def test_equal_lengths(l_t, n_layers):
    check_encoder(shape(l_t, n_layers))


@pytest.mark.parametrize("l_t", [5, 40, 140])
def test_many_lengths(l_t):
    s = shape(l_t, 2)
    check_encoder(s, synth.item_lengths(3, s.n_items, l_t, 1))


def test_more_items_than_blocks():
    check_encoder(shape(3, 1, n_items=1300))
