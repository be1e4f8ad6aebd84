"""Sample sort of the survivors (KMER_FLAG_SORTED_OUTPUT) at the sizes where its steps change: one bucket, one and
two levels of splitters, key widths one to four, tallies past 16 bits, and thousands of keys alike in their first
64 bits (the digit-by-digit sort takes over).  The reference is the unsorted result of the same reads, ordered on
the host.  Everything is integer: the comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)


def both(reads, k, **params):
    """(sorted result, unsorted result ordered on the host, stats of the sorted query)"""
    import paper_1809_07014_gb300 as km
    bases = np.ascontiguousarray(np.concatenate(reads))
    quals = np.full(len(bases), 33 + 40, dtype=np.uint8)
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    rs = km.ReadSet(bases, quals, offsets)
    out = []
    for flags in (km.KMER_FLAG_SORTED_OUTPUT, 0):
        ka = km.KmerAnalysis(k, flags=flags, **params)
        ka.submit(rs)
        out.append(ka.results())
        st = ka.stats() if flags else st
        ka.close()
    got, want = out
    order = np.lexsort([want.keys[:, w] for w in reversed(range(want.keys.shape[1]))])
    rs.close()
    return got, want, order, st


def check(got, want, order):
    assert got.windows == want.windows and got.distinct == want.distinct
    np.testing.assert_array_equal(got.keys, want.keys[order])
    np.testing.assert_array_equal(got.count, want.count[order])
    np.testing.assert_array_equal(got.ext, want.ext[order])
    np.testing.assert_array_equal(got.cls, want.cls[order])


# one bucket (up to 1024), one level (up to 589 824), two levels
@pytest.mark.parametrize("k", [9, 31, 33, 63, 77, 127])
@pytest.mark.parametrize("n", [2, 1024, 1025, 40_003, 589_824, 589_825, 1_500_001])
def test_sizes(k, n):
    rng = np.random.default_rng(n + k)
    if k == 9 and n > 100_000:
        pytest.skip("4^9 / 2 k-mers at most")
    genome = LETTERS[rng.integers(0, 4, n + k - 1)]  # n windows, nearly all distinct for k > 9
    step = 4000
    reads = [genome[i:min(i + step, n) + k - 1] for i in range(0, n, step)]
    got, want, order, st = both(reads, k, min_count=1)
    if k > 9:
        assert len(got.count) == n
    assert st["n_sort"] == 0
    check(got, want, order)


def test_wide_tallies():
    rng = np.random.default_rng(5)
    hot = LETTERS[rng.integers(0, 4, 40)]
    reads = [hot] * 70_000 + [LETTERS[rng.integers(0, 4, 150)] for _ in range(2000)]
    for k in (31, 33):
        got, want, order, _ = both(reads, k, min_count=1)
        assert got.ext.max() >= 65536
        check(got, want, order)


@pytest.mark.parametrize("k", [63, 127])
def test_alike_in_the_first_64_bits(k):
    # 20 000 k-mers that begin with the same 32 A: more than one CTA sorts
    rng = np.random.default_rng(k)
    reads = [np.concatenate([np.full(32, ord("A"), np.uint8), LETTERS[rng.integers(0, 4, k - 32)]])
             for _ in range(20_000)]
    got, want, order, st = both(reads, k, min_count=1)
    assert len(got.count) > 19_000
    check(got, want, order)


def test_clusters():
    # a deep amplicon: every k-mer has hundreds of neighbours alike in their first half
    rng = np.random.default_rng(9)
    amp = LETTERS[rng.integers(0, 4, 150)]
    reads = []
    for _ in range(30_000):
        r = amp.copy()
        at = rng.integers(0, 150, 3)
        r[at] = LETTERS[rng.integers(0, 4, 3)]
        reads.append(r)
    for k in (31, 55):
        got, want, order, _ = both(reads, k, min_count=1)
        check(got, want, order)
