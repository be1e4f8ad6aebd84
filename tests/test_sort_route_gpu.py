"""Which sort orders the survivors: one timed sort for the sample sort alone, two when the sort by digits takes over
because more keys than one CTA sorts begin with the same 64 bits.  The order itself is checked on the host."""
import numpy as np
import pytest

from tests.test_sample_sort_gpu import LETTERS

pytestmark = pytest.mark.gpu


def sorts(reads, k):
    import paper_1809_07014_gb300 as km
    bases = np.ascontiguousarray(np.concatenate(reads))
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    rs = km.ReadSet(bases, np.full(len(bases), 33 + 40, np.uint8), offsets)
    ka = km.KmerAnalysis(k, min_count=1, flags=km.KMER_FLAG_SORTED_OUTPUT | km.KMER_FLAG_PROFILE)
    ka.submit(rs)
    res, st = ka.results(), ka.stats()
    ka.close()
    rs.close()
    order = np.lexsort([res.keys[:, w] for w in reversed(range(res.keys.shape[1]))])
    np.testing.assert_array_equal(order, np.arange(len(order)))
    return st["n_sort"]


@pytest.mark.parametrize("k", [31, 33, 77, 127])
@pytest.mark.parametrize("n", [1000, 40_003, 1_500_001])
def test_random_keys_take_the_sample_sort(k, n):
    rng = np.random.default_rng(n + k)
    genome = LETTERS[rng.integers(0, 4, n + k - 1)]
    assert sorts([genome[i:min(i + 4000, n) + k - 1] for i in range(0, n, 4000)], k) == 1


def test_clusters_take_the_sample_sort():
    rng = np.random.default_rng(9)
    amp = LETTERS[rng.integers(0, 4, 150)]
    reads = []
    for _ in range(30_000):
        r = amp.copy()
        at = rng.integers(0, 150, 3)
        r[at] = LETTERS[rng.integers(0, 4, 3)]
        reads.append(r)
    assert sorts(reads, 31) == 1


@pytest.mark.parametrize("k", [63, 127])
def test_alike_keys_take_the_sort_by_digits(k):
    rng = np.random.default_rng(k)
    reads = [np.concatenate([np.full(32, ord("A"), np.uint8), LETTERS[rng.integers(0, 4, k - 32)]])
             for _ in range(20_000)]
    assert sorts(reads, k) == 2
