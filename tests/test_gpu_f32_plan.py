"""fp32 contexts whose products lie at the lines of the plan that cuts a K range: two, four and eight parts of one round of four groups,
with remainders, and the sizes just beside them that keep more parts."""
import pytest

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests import gram_helpers as gh

pytestmark = pytest.mark.gpu

BASE = dict(dtype="f32", vocab=40, pooling="mean", task="kt", task_layers=1, task_heads=2, task_attn_only=False, zipf_s=0.5, n_items=12, l_t=3,
            n_layers=1, n_heads=2, d_ff=32)
SHAPES = {                                                    # the second product of the task's feed-forward, rows x d over task_d_ff
    "912x64x256_two": dict(d=64, task_d_ff=256, B=8, L=114),
    "480x64x384_four": dict(d=64, task_d_ff=384, B=5, L=96),
    "912x32x1024_eight": dict(d=32, task_d_ff=1024, B=8, L=114),
    "903x28x1000_eight": dict(d=28, task_d_ff=1000, B=21, L=43),
    "1760x32x256_two": dict(d=32, task_d_ff=256, B=16, L=110),
    "1600x32x256_more": dict(d=32, task_d_ff=256, B=16, L=100),
    "576x128x384_more": dict(d=128, task_d_ff=384, B=6, L=96),
    "160x64x256_more": dict(d=64, task_d_ff=256, B=2, L=80),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_products_at_the_lines(name):
    shape = synth.GramShape(**{**BASE, "name": name, **SHAPES[name]})
    ce, tk, toks, ids, lab = gh.make_inputs(shape, seed=9)
    want = orc.gram_single_step(shape, ce, tk, toks, ids, lab)
    rep, gce, gtk = gh.gpu_single_step(shape, ce, tk, toks, ids, lab)
    # fp32 sums against 64 bits: 2e-6 is what such models show on their worst tensor; an order of magnitude above it
    assert abs(rep.loss - want["loss"]) <= 2e-5 * abs(want["loss"])
    assert gh.worst_rel_err(gce, want["grad_ce"])[0] <= 2e-5
    assert gh.worst_rel_err(gtk, want["grad_task"])[0] <= 2e-5
