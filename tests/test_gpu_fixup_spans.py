"""Segment sums of items that reach over the ends of their chunks by as many chunks as one warp adds up alone, one more, and twice as
many: 1600 positions are 100 chunks of 16."""
import numpy as np
import pytest
import torch

from tests.test_gpu_index import index_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [4, 128, 260, 768])
@pytest.mark.parametrize("chunks", [1, 4, 5, 8, 9, 16, 17, 99])
def test_items_over_many_chunks(d, chunks):
    P = 1600
    # an item that begins in the middle of chunk 0 and ends in the middle of chunk `chunks`, short ones before and behind
    seg = np.unique(np.concatenate([[0, 3, 7, 16 * chunks + (8 if chunks < 99 else 16)], np.arange(16 * chunks + 8, P + 1, 5), [P]])).astype(np.int32)
    U = len(seg) - 1
    g = index_ctx(P, U, d)
    gen = torch.Generator().manual_seed(chunks)
    dE = (torch.rand(P, d, generator=gen) * 2 - 1).cuda()
    perm = torch.randperm(P, generator=gen).to(torch.int32).cuda()
    G = torch.full((U, d), -7.0, device="cuda")
    g.accumulate(dE, perm, torch.from_numpy(seg).cuda(), U, G)
    g.sync()
    g.close()
    rows = dE[perm.long()].double()
    for u in range(U):
        n = int(seg[u + 1] - seg[u])
        want = rows[seg[u]:seg[u + 1]].sum(0)
        # n terms of at most 1: n - 1 additions of sums below n, each rounded once
        assert (G[u] - want).abs().max() <= n * 2.0 ** -24 * n + 1e-6, u
