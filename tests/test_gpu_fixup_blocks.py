"""Segment sums on both sides of the line where the fix-up of items over chunk ends takes eight chunks to a block instead of one: the most
(chunk, slab) pairs that go one to a block, and the next size.  Items end in the middle and at the ends of chunks, over one to forty of them."""
import numpy as np
import pytest
import torch

from tests.test_gpu_index import index_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,d", [(18_944, 128), (18_960, 128), (6304, 768), (6320, 768), (6336, 700)])     # 1184, 1185, 1182, 1185, 1188 pairs
@pytest.mark.parametrize("table", [False, True])
def test_items_over_chunk_ends(P, d, table):
    gen = np.random.default_rng(P + d)
    lengths = []
    while sum(lengths) < P:                                   # chunks of 16 positions: an item of 16 k + r reaches over k or k + 1 chunk ends
        k = int(gen.choice([0, 0, 0, 1, 7, 8, 9, 10, 16, 17, 18, 40]))
        lengths.append(max(1, 16 * k + int(gen.choice([0, 3, 8]))))
    seg = np.minimum(np.concatenate([[0], np.cumsum(lengths)]), P).astype(np.int32)
    U = len(seg) - 1
    dE = torch.rand(P, d, generator=torch.Generator().manual_seed(d)).cuda() * 2 - 1
    perm = torch.from_numpy(gen.permutation(P).astype(np.int32)).cuda()
    s = torch.from_numpy(seg).cuda()
    item = torch.repeat_interleave(torch.arange(U, device="cuda"), torch.diff(s.long()))
    x = dE[perm.long()].double()
    g = index_ctx(P, max(P, 2 * U), d)
    if table:
        rows = torch.from_numpy(gen.permutation(2 * U)[:U].astype(np.int32)).cuda()
        old = torch.randn(2 * U, d, device="cuda")
        out = old.clone()
        bits = torch.zeros((2 * U + 31) // 32, dtype=torch.int32, device="cuda")
        g.accumulate_multistep(dE, perm, s, rows, U, 2 * U, out, bits)
        want, size = old[rows.long()].double(), old[rows.long()].double().abs()
    else:
        out = torch.full((U, d), float("nan"), device="cuda")
        g.accumulate(dE, perm, s, U, out)
        want = torch.zeros(U, d, dtype=torch.float64, device="cuda")
        size = torch.zeros_like(want)
    g.sync()
    g.close()
    want.index_add_(0, item, x)
    size.index_add_(0, item, x.abs())
    got = out[rows.long()] if table else out
    # a sum is a chain of at most one chunk's rows, then of five parts, then of eight runs, then the old value: 2^-24 of what has been added for
    # each link
    assert ((got.double() - want).abs() <= (16 + 5 + 8 + 1) * 2.0 ** -24 * size + 1e-6).all()
    if table:
        rest = torch.ones(2 * U, dtype=torch.bool, device="cuda")
        rest[rows.long()] = False
        assert torch.equal(out[rest], old[rest])
