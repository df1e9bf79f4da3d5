"""fp32 contexts at the edges of the launch that takes a gradient's two products together: remainders in every
direction, one row, long sums over few tiles, the last size that goes together and the first that does not, small clusters."""
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu

BASE = dict(dtype="f32", vocab=40, pooling="mean", task="kt", task_layers=1, task_attn_only=False, zipf_s=0.5, n_items=12, l_t=3, n_layers=1)
SHAPES = {
    "one_position": dict(d=32, n_heads=2, d_ff=32, B=1, L=1, task_heads=2, task_d_ff=32),
    "remainders": dict(d=36, n_heads=2, d_ff=68, B=7, L=19, task_heads=2, task_d_ff=100, l_t=11),
    "attention_only": dict(d=44, n_heads=2, d_ff=68, B=9, L=21, task_heads=2, task_d_ff=68, task_attn_only=True, task_layers=2),
    # one tile of dW over 5000 rows: sixteen parts of it beside tiles of dX in one part
    "long_sum": dict(d=16, n_heads=1, d_ff=32, B=50, L=100, task_heads=1, task_d_ff=32),
    # 8 + 4 * 109 = 444 tiles in the first product of the feed-forward's backward pass, 8 + 4 * 110 in the second shape
    "last_together": dict(d=64, n_heads=2, d_ff=64, B=32, L=109, task_heads=2, task_d_ff=128),
    "first_apart": dict(d=64, n_heads=2, d_ff=64, B=33, L=106, task_heads=2, task_d_ff=128),
}


def check(shape, clusters):
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=7)
    want = orc.gram_single_step(shape, ce, tk, toks, ids, lab)
    g = gh.make_ctx(shape, ce, tk, toks)
    if clusters:
        g.selftest_cluster_blocks(clusters)
    rep = g.step(torch.from_numpy(ids).cuda(), torch.from_numpy(lab).cuda(), ids.shape[0])
    gce, gtk = gh.gpu_grads(g, shape)
    g.close()
    # fp32 sums against 64 bits: 2e-6 is what such models show on their worst tensor; an order of magnitude above it
    assert abs(rep.loss - want["loss"]) <= 2e-5 * abs(want["loss"])
    assert gh.worst_rel_err(gce, want["grad_ce"])[0] <= 2e-5
    assert gh.worst_rel_err(gtk, want["grad_task"])[0] <= 2e-5


@pytest.mark.parametrize("name", list(SHAPES))
def test_gradient_products_together(name):
    check(synth.GramShape(**{**BASE, "name": name, **SHAPES[name]}), 0)


@pytest.mark.parametrize("clusters", [1, 2, 8])
def test_gradient_products_in_small_clusters(clusters):
    check(synth.GramShape(**{**BASE, "name": "c", **SHAPES["remainders"]}), clusters)
