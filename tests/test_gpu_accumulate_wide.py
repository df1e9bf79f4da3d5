"""Segment sums of wide rows on both sides of the lines where the kernel changes, against 64-bit sums: last chunks that are
short, one item for all positions, every position its own item."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests.test_gpu_index import index_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["zipf", "one", "distinct"])
@pytest.mark.parametrize("P,d", [(19_999, 768), (20_000, 516), (20_001, 768), (37_889, 768), (50_003, 1024), (75_777, 512), (75_777, 600)])
def test_segment_sums_of_wide_rows(P, d, kind):
    ids = {"zipf": lambda: synth.zipf_ids(3, 5000, 1.0, P), "one": lambda: np.zeros(P, np.int32),
           "distinct": lambda: np.random.default_rng(1).permutation(P).astype(np.int32)}[kind]()
    unique, _, perm, seg = orc.unique_inverse(ids)
    U = len(unique)
    dE = torch.rand(P, d, generator=torch.Generator().manual_seed(P + d)) * 2 - 1
    g = index_ctx(P, max(P, 5000), d)
    p, s = torch.from_numpy(perm.astype(np.int32)).cuda(), torch.from_numpy(seg.astype(np.int32)).cuda()
    x = dE.cuda()
    out = [torch.full((U, d), float("nan"), device="cuda") for _ in range(2)]
    for o in out:
        g.accumulate(x, p, s, U, o)
    g.sync()
    g.close()
    assert torch.equal(out[0], out[1])                        # bit-identical from call to call
    want = torch.zeros(U, d, dtype=torch.float64, device="cuda")
    size = torch.zeros_like(want)
    item = torch.repeat_interleave(torch.arange(U, device="cuda"), torch.diff(s.long()))
    want.index_add_(0, item, x[p.long()].double())
    size.index_add_(0, item, x[p.long()].double().abs())
    # a sum is a chain of at most one chunk's rows, then of an eighth of the chunks' parts, then of eight: 2^-24 of what has
    # been added for each link (for one item of 50 003 rows 0.5, where a chunk's part is about 3)
    chunks = min(-(-P // 16), 148 * 16)
    links = -(-P // chunks) + -(-chunks // 8) + 8
    assert ((out[0].double() - want).abs() <= links * 2.0 ** -24 * size + 1e-6).all()
