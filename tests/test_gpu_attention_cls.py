"""Token-0 pooling with heads of width 64: the last layer's attention runs with one query row per item."""
import os
import subprocess
import sys

import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh
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


@pytest.mark.parametrize("heads", [4, 13])
@pytest.mark.parametrize("l_t", [16, 23, 24, 33])
def test_encodings_on_both_sides_of_the_forward_kernel_s_line(l_t, heads):
    """Texts that fetch as they go and texts that fetch ahead, with the registers of up to twelve and of up to sixteen heads."""
    s = shape(l_t, 1).replace(d=64 * heads, n_heads=heads)
    # weights such that sums over the width vary as check_encoder's do over 128 columns at 0.1, whose bound this takes over
    ce, tk, toks, _, _ = gh.make_inputs(s, seed=6, sigma=0.1 * (128 / s.d) ** 0.5)
    lengths = synth.item_lengths(3, s.n_items, l_t, 1)
    for texts, given in ((toks, None), (synth.ragged(toks, lengths), lengths)):
        g = gh.make_ctx(s, ce, tk, toks)
        if given is not None:
            g.set_item_lengths(given)
        H = torch.empty(s.n_items, s.d, device="cuda")
        g.encode_unique(None, torch.arange(s.n_items, dtype=torch.int32, device="cuda"), s.n_items, H)
        g.sync()
        g.close()
        th = orc.as_torch(ce)
        want = torch.stack([orc.ce_forward(th, texts[i], s) for i in range(s.n_items)])
        assert gh.rel_err(H.cpu().numpy(), want.detach().numpy()) <= 2e-2            # bf16 operands, as in check_encoder


def test_more_items_than_blocks():
    check_encoder(shape(3, 1, n_items=1300))


CHILD = """
import torch
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh
from tests.test_gpu_attention_cls import shape
s = shape(20, 1)
ce, tk, toks, _, _ = gh.make_inputs(s, seed=6)
g = gh.make_ctx(s, ce, tk, toks)
g.profile(True)
g.encode_unique(None, torch.arange(s.n_items, dtype=torch.int32, device="cuda"), s.n_items, torch.empty(s.n_items, s.d, device="cuda"))
g.sync()
print(" ".join(sorted(g.profile_dump())))
"""


@pytest.mark.parametrize("forced", [False, True])
def test_the_switch_that_forces_the_tcgen05_kernels(forced):
    """GRAM_ATTN_TC=1 (read once per process) leaves no attention to other kernels, the last layer's included."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = {k: v for k, v in os.environ.items() if k != "GRAM_ATTN_TC"}
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=root, env=dict(env, GRAM_ATTN_TC="1") if forced else env, capture_output=True,
                         text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-1000:]
    tags = out.stdout.split()
    assert ("attn_cls_fwd" in tags, "attn_fwd" in tags) == (not forced, forced)
