"""fp32 contexts at sizes that reach every form of the fp32 matrix product: 32- and 64-wide tiles, the K range in one
piece and over clusters of up to 16 blocks, rows that allow 16-byte loads and rows that do not."""
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu

SHAPES = {
    # rows of 18 floats (attention pooling, news task): no 16-byte loads; about 2000 token rows: weight gradients over 16 parts
    "odd_rows": dict(d=12, n_heads=1, d_ff=16, l_t=9, n_items=260, B=30, L=12, pooling="additive", d_a=18, task="nr", task_layers=0,
                     n_cand=3),
    # 64-wide tiles in the forward products, remainders in rows and columns
    "large_tiles": dict(d=72, n_heads=2, d_ff=264, l_t=17, n_items=420, B=40, L=20, task_heads=2, task_d_ff=136, n_layers=1),
    # widths 32, 64 and 128 over some 900, 1600 and 1200 token rows: one round of two and of four groups, eight parts of four groups,
    # sixteen parts of one, K ranges that leave groups of the last round without a k-block
    "width_32": dict(d=32, n_heads=2, d_ff=128, l_t=15, n_items=60, B=8, L=20, task_heads=2, task_d_ff=128, n_layers=1),
    "width_64": dict(d=64, n_heads=2, d_ff=256, l_t=16, n_items=100, B=30, L=20, task_heads=2, task_d_ff=256, n_layers=1),
    "width_128": dict(d=128, n_heads=2, d_ff=512, l_t=15, n_items=80, B=8, L=20, task_heads=2, task_d_ff=512, n_layers=1),
    # 304 tiles and K = 1024: groups without parts
    "width_256": dict(d=256, n_heads=4, d_ff=1024, l_t=15, n_items=80, B=30, L=20, task_heads=4, task_d_ff=1024, n_layers=1),
    "one_row": dict(d=32, n_heads=2, d_ff=64, l_t=1, n_items=1, B=1, L=1, task_heads=2, task_d_ff=64),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_f32_step(name):
    shape = synth.GramShape(**dict(dict(name=name, dtype="f32", vocab=50, pooling="mean", task="kt", task_layers=1, task_attn_only=False,
                                        zipf_s=0.5), **SHAPES[name]))
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=4)
    want = orc.gram_single_step(shape, ce, tk, toks, ids, lab)
    rep, gce, gtk = gh.gpu_single_step(shape, ce, tk, toks, ids, lab)
    # fp32 sums against 64 bits: 2e-6 is what such models show on their worst tensor; an order of magnitude above it
    assert abs(rep.loss - want["loss"]) <= 2e-5 * abs(want["loss"])
    assert gh.worst_rel_err(gce, want["grad_ce"])[0] <= 2e-5
    assert gh.worst_rel_err(gtk, want["grad_task"])[0] <= 2e-5


@pytest.mark.parametrize("blocks", [8, 1])
def test_f32_step_where_smaller_clusters_are_placed(blocks):
    shape = synth.GramShape(**dict(dict(name="c", dtype="f32", vocab=50, pooling="mean", task="kt", task_layers=1, task_attn_only=False,
                                        zipf_s=0.5), **SHAPES["odd_rows"]))
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=4)
    want = orc.gram_single_step(shape, ce, tk, toks, ids, lab)
    g = gh.make_ctx(shape, ce, tk, toks)
    g.selftest_cluster_blocks(blocks)
    rep = g.step(torch.from_numpy(ids).cuda(), torch.from_numpy(lab).cuda(), ids.shape[0])
    gce, gtk = gh.gpu_grads(g, shape)
    g.close()
    assert abs(rep.loss - want["loss"]) <= 2e-5 * abs(want["loss"])
    assert gh.worst_rel_err(gce, want["grad_ce"])[0] <= 2e-5
    assert gh.worst_rel_err(gtk, want["grad_task"])[0] <= 2e-5
