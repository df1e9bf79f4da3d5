"""Segment sums added to picked rows of a table, against 64-bit sums: chunks of 33 to 100 positions, so that a chunk goes through more than
the 32 items (twice as many, one more, three times and some) whose ends and rows its warp holds at a time; by the chunks kernel and by
both widths of the ring kernel."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests.test_gpu_index import index_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["distinct", "zipf"])
@pytest.mark.parametrize("P", [75_777, 149_185, 151_553, 234_433])
@pytest.mark.parametrize("d", [64, 260, 600, 1024])
def test_sums_into_a_table(P, d, kind):
    gen = torch.Generator().manual_seed(P + d)
    if kind == "distinct":
        U = P
        perm, seg = torch.randperm(P, generator=gen, dtype=torch.int64), torch.arange(P + 1)
    else:
        unique, _, perm, seg = orc.unique_inverse(synth.zipf_ids(3, 60_000, 0.8, P))
        U, perm, seg = len(unique), torch.from_numpy(np.asarray(perm, np.int64)), torch.from_numpy(np.asarray(seg, np.int64))
    N = U + U // 3
    rows = torch.randperm(N, generator=gen)[:U]
    perm, seg, rows = perm.cuda(), seg.cuda(), rows.cuda()
    cgen = torch.Generator(device="cuda").manual_seed(P + d)
    dE = torch.rand(P, d, generator=cgen, device="cuda") * 2 - 1
    start = torch.randn(N, d, generator=cgen, device="cuda")
    g = index_ctx(P, N, d)
    tables = [start.clone() for _ in range(2)]
    bits = torch.zeros((N + 31) // 32, dtype=torch.int32, device="cuda")
    for t in tables:
        g.accumulate_multistep(dE, perm.int(), seg.int(), rows.int(), U, N, t, bits)
    g.sync()
    g.close()
    assert torch.equal(tables[0], tables[1])                  # bit-identical from call to call
    rest = torch.ones(N, dtype=torch.bool, device="cuda")
    rest[rows] = False
    assert torch.equal(tables[0][rest], start[rest])
    touched = (bits[:, None] >> torch.arange(32, device="cuda", dtype=torch.int32) & 1).bool().flatten()[:N]
    assert torch.equal(touched, ~rest)
    # a sum is a chain of at most one chunk's rows, then of an eighth of the chunks' parts, then of eight, then the old value: 2^-24 of
    # what has been added for each link
    links = -(-P // 2368) + 2368 // 8 + 8 + 1
    item = torch.repeat_interleave(torch.arange(U, device="cuda"), torch.diff(seg))
    for c in range(0, d, 256):                                # columns in slabs: 64-bit copies of all would not be small
        x = dE[:, c:c + 256][perm].double()
        want = start[rows][:, c:c + 256].double()
        size = want.abs()
        want.index_add_(0, item, x)
        size.index_add_(0, item, x.abs())
        assert ((tables[0][rows][:, c:c + 256].double() - want).abs() <= links * 2.0 ** -24 * size + 1e-6).all()
