"""Hundreds of leaves that overflow their tables one after another on every CTA: each warp has to see the overflow before
it is cleared for the next leaf, or it writes a part of a half-counted table.  The reference is the same query in
leaves that fit.  Everything is integer: the comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)


@pytest.mark.parametrize("k", [31, 55, 77, 127])
def test_overfull_leaves(k):
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(k)
    n, step = 3_000_000, 2000
    genome = LETTERS[rng.integers(0, 4, n + k)]
    reads = [genome[i:i + step + k - 1] for i in range(0, n, step)]
    bases = np.concatenate(reads)
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    rs = km.ReadSet(bases, np.full(len(bases), 33 + 40, np.uint8), offsets)

    def run(leaf_bits):
        ka = km.KmerAnalysis(k, min_count=1, flags=km.KMER_FLAG_SORTED_OUTPUT, leaf_bits=leaf_bits)
        ka.submit(rs)
        out = [ka.results(ka.query()) for _ in range(1 if leaf_bits == 12 else 5)], ka.stats()
        ka.close()
        return out

    (want,), st = run(12)
    assert st["leaf_splits"] == 0
    got, st = run(9)  # 5860 keys a leaf: two tables and more
    assert st["leaf_splits"] > 400, st
    for r in got:
        assert r.windows == want.windows and r.distinct == want.distinct
        np.testing.assert_array_equal(r.keys, want.keys)
        np.testing.assert_array_equal(r.count, want.count)
        np.testing.assert_array_equal(r.ext, want.ext)
        np.testing.assert_array_equal(r.cls, want.cls)
    rs.close()
