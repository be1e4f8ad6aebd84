"""Leaf tables from nearly empty to overfull: forced leaf counts put a tenth of a table to several tables of keys in
each leaf (the latter counted in key ranges), with every key seen once or many times.  Compared with the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)


@pytest.mark.parametrize("k", [21, 31, 33, 63, 77, 127])
@pytest.mark.parametrize("leaf_bits", [7, 5, 4, 3])
def test_loads(k, leaf_bits):
    import oracle
    import paper_1809_07014_gb300 as km
    from tests.helpers import assert_same

    rng = np.random.default_rng(1000 * leaf_bits + k)
    once = LETTERS[rng.integers(0, 4, 30_000 + k)]
    often = LETTERS[rng.integers(0, 4, 2_000 + k)]
    reads = [once[i:i + 500 + k - 1] for i in range(0, 30_000, 500)]
    for _ in range(40):
        i = int(rng.integers(0, 1500))
        reads.append(often[i:i + 500 + k - 1])
    bases = np.concatenate(reads)
    quals = rng.integers(33 + 10, 33 + 41, len(bases)).astype(np.uint8)
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    rs = km.ReadSet(bases, quals, offsets)
    for min_count in (1, 2):
        want = oracle.run(bases, quals, offsets, oracle.Params(k=k, min_count=min_count))
        ka = km.KmerAnalysis(k, min_count=min_count, leaf_bits=leaf_bits)
        ka.submit(rs)
        for _ in range(2):  # the second query sizes its tables from the first
            assert_same(ka.results(ka.query()), want, f"k={k} leaf_bits={leaf_bits} min_count={min_count}")
        ka.close()
    rs.close()
