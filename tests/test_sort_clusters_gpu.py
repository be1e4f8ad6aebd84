"""Sorted output of k-mers that begin alike in clusters: ranges of a bucket that hold more keys than they are counted in
go through a sorting network.  The reference is the unsorted result ordered on the host (exact); clusters must not
take many times what random keys take."""
import numpy as np
import pytest

from tests.test_lookup_stream_gpu import LETTERS

pytestmark = pytest.mark.gpu


def readset(k, shared, cluster, n, rng):
    # every read is one k-mer that starts and ends with A, so that it is its own canonical form
    import paper_1809_07014_gb300 as km
    heads = np.repeat(rng.integers(0, 4, (-(-n // cluster), shared), dtype=np.uint8), cluster, axis=0)[:n]
    tails = rng.integers(0, 4, (n, k - shared), dtype=np.uint8)
    heads[:, 0] = tails[:, -1] = 0
    bases = LETTERS[np.concatenate([heads, tails], axis=1)].reshape(-1)
    return km.ReadSet(bases, np.full(len(bases), 73, np.uint8), np.arange(n + 1, dtype=np.uint64) * np.uint64(k))


def query(rs, k, flags):
    import paper_1809_07014_gb300 as km
    ka = km.KmerAnalysis(k, min_count=1, flags=flags)
    ka.submit(rs)
    res = ka.results()
    for _ in range(3):
        ka.query()
    st = ka.stats()
    ka.close()
    return res, st


# one bucket, one level and two levels of splitters; ranges below, at and above the lines of 32 and 128
@pytest.mark.parametrize("k, shared", [(31, 12), (31, 26), (33, 32), (55, 32), (77, 40), (127, 33), (127, 110)])
@pytest.mark.parametrize("n, cluster", [(2, 2), (1000, 1000), (1024, 31), (3000, 33), (50_000, 129), (50_000, 1200),
                                        (700_000, 700), (700_000, 40)])
def test_order(k, shared, n, cluster):
    import paper_1809_07014_gb300 as km
    rs = readset(k, shared, cluster, n, np.random.default_rng(n + cluster + k))
    got, _ = query(rs, k, km.KMER_FLAG_SORTED_OUTPUT)
    want, _ = query(rs, k, 0)
    order = np.lexsort([want.keys[:, w] for w in reversed(range(want.keys.shape[1]))])
    for c in ("keys", "count", "ext", "cls"):
        np.testing.assert_array_equal(getattr(got, c), getattr(want, c)[order])
    rs.close()


@pytest.mark.parametrize("k, shared", [(31, 16), (55, 32), (127, 32)])
def test_clusters_cost_little(k, shared):
    import paper_1809_07014_gb300 as km
    took = {}
    for cluster in (1, 400):
        rs = readset(k, shared, cluster, 2_000_000, np.random.default_rng(k))
        st = query(rs, k, km.KMER_FLAG_SORTED_OUTPUT | km.KMER_FLAG_PROFILE)[1]
        assert st["n_sort"] == 1
        took[cluster] = st["ms_sort"]
        rs.close()
    assert took[400] < 5 * took[1], took  # counting took 17 times as long at k = 55
