"""gram_dedup at the edges of its one-launch form: the tiles of one thread block, full clusters, one position more."""
import numpy as np
import pytest

from oracle import gram_oracle as orc
from paper_2204_04179_b200 import synth
from tests.test_gpu_index import index_ctx, run_dedup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["zipf", "same", "descending"])
@pytest.mark.parametrize("P", [2, 511, 513, 8192, 8193, 16_385, 65_537, 131_071, 131_072, 131_073])
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
