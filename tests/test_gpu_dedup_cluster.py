"""gram_dedup at the edges of its one-launch form (the tiles of one thread block, full clusters, one position more) and of the
chain of launches: one, two and three passes, the last tile full, one key short, one key long."""
import numpy as np
import pytest
import torch

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import binding, synth
from tests.test_gpu_index import index_ctx, run_dedup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["zipf", "same", "descending"])
@pytest.mark.parametrize("P", [2, 511, 513, 8192, 8193, 16_385, 32_768, 32_769, 40_001, 65_535, 65_536, 65_537, 131_072, 131_073])
def test_dedup_at_tile_and_cluster_edges(P, kind):
    n = {"zipf": 70_001, "same": 300, "descending": P}[kind]
    ids = {"zipf": lambda: synth.zipf_ids(5, n, 1.0, P), "same": lambda: np.full(P, n - 1, np.int32),
           "descending": lambda: np.arange(P - 1, -1, -1, dtype=np.int32)}[kind]()
    g = index_ctx(P, n, 4)
    U, *got = run_dedup(g, ids, n)
    want = orc.unique_inverse(ids)
    assert U == len(want[0])
    for x, w in zip(got, want):                          # whole numbers: one correct answer
        assert np.array_equal(x, w)
    g.close()


@pytest.mark.parametrize("n_items", [1, 2, 300, 1024, 1025, 65_536, 1_048_576, 1_048_577, 20_000_000])
@pytest.mark.parametrize("P", [65_537, 73_728, 73_729, 524_288 + 8191])
def test_dedup_chain_of_launches(P, n_items):
    ids = synth.zipf_ids(6, n_items, 0.9, P)
    ids[: min(P, 50)] = n_items - 1                      # the largest key that the passes must place
    g = index_ctx(P, n_items, 4)
    U, *got = run_dedup(g, ids, n_items)
    want = orc.unique_inverse(ids)
    assert U == len(want[0])
    for x, w in zip(got, want):
        assert np.array_equal(x, w)
    g.close()


@pytest.mark.parametrize("kind", ["half", "same", "two", "runs", "uniform"])
@pytest.mark.parametrize("n_items", [100, 40_000, 200_000, 900_000])
def test_dedup_of_one_id_that_fills_the_batch(n_items, kind):
    """Passes of 7 to 10 bits over rounds of 32 keys of which all, half, some or one have the first key's digit; the last
    tile ends inside a round."""
    P = 73_728 + 32 * 20 + 5
    rng = np.random.default_rng(n_items)
    ids = rng.integers(0, n_items, P).astype(np.int32)
    if kind == "half":
        ids[rng.random(P) < 0.5] = n_items - 1
    elif kind == "same":
        ids[:] = n_items // 2
    elif kind == "two":
        ids = np.where(ids % 2 == 0, 1, n_items - 2).astype(np.int32)
    elif kind == "runs":
        ids = np.repeat(ids, rng.integers(1, 60, P))[:P].copy()
    g = index_ctx(P, n_items, 4)
    U, *got = run_dedup(g, ids, n_items)
    want = orc.unique_inverse(ids)
    assert U == len(want[0])
    for x, w in zip(got, want):
        assert np.array_equal(x, w)
    g.close()


def test_dedup_of_fewer_items_than_the_context_holds():
    """A context for many items serves calls with any number of them: the widths of the passes differ from call to call."""
    P = 200_000
    g = index_ctx(P, 20_000_000, 4)
    for n_items in (20_000_000, 900_000, 5000, 700, 3, 1_100_000):
        ids = synth.zipf_ids(7, n_items, 1.0, P)
        U, *got = run_dedup(g, ids, n_items)
        want = orc.unique_inverse(ids)
        assert U == len(want[0])
        for x, w in zip(got, want):
            assert np.array_equal(x, w)
    g.close()


@pytest.mark.parametrize("blocks", [8, 4, 2, 1])
def test_dedup_where_smaller_clusters_are_placed(blocks):
    """A process limited to part of the multiprocessors: the one-launch form up to 4096 positions per block that can be placed,
    the chain of launches beyond, also for contexts of few positions."""
    for P in (3, 4096, 4097, 8192, 25_600, 32_768, 32_769, 65_536):
        ids = synth.zipf_ids(8, 10_000, 1.0, P)
        g = index_ctx(P, 10_000, 4)
        g.selftest_cluster_blocks(blocks)
        U, *got = run_dedup(g, ids, 10_000)
        want = orc.unique_inverse(ids)
        assert U == len(want[0])
        for x, w in zip(got, want):
            assert np.array_equal(x, w)
        g.close()


@pytest.mark.parametrize("P", [700, 9000, 40_000, 65_537])
def test_ids_out_of_range(P):
    """Both forms report the error, sort such an ID as item 0 and give its positions the index -1."""
    n = 500
    ids = synth.zipf_ids(9, n, 1.0, P)
    ids[::97] = n
    ids[5::131] = -3
    bad = (ids < 0) | (ids >= n)
    unique, inverse, perm, seg = orc.unique_inverse(np.where(bad, 0, ids).astype(np.int32))
    g = index_ctx(P, n, 4)
    out = [torch.zeros(k, dtype=torch.int32, device="cuda") for k in (n, P, P, n + 1, 1)]
    g.dedup(torch.from_numpy(ids).cuda(), n, *out)
    with pytest.raises(binding.GramError, match="GRAM_ERR_ID_RANGE"):
        g.sync()
    U = int(out[4].item())
    assert U == len(unique) and np.array_equal(out[0][:U].cpu().numpy(), unique)
    assert np.array_equal(out[1].cpu().numpy(), np.where(bad, -1, inverse))
    assert np.array_equal(out[2].cpu().numpy(), perm) and np.array_equal(out[3][:U + 1].cpu().numpy(), seg)
    g.close()
