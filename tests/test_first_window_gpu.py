"""The first window of a read is taken from the packed blocks at once: reads of length k - 1 .. k + 66 with an N, or a
low-quality base, at each edge of the first window and of the 32-base blocks around it.  Compared with the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("k", [1, 15, 17, 31, 33, 63, 65, 95, 97, 127])
def test_edges(k, variant):
    import oracle
    import paper_1809_07014_gb300 as km
    from tests.helpers import assert_same

    rng = np.random.default_rng(k)
    genome = LETTERS[rng.integers(0, 4, 400)]
    reads, quals = [], []
    for length in {k - 1, k, k + 1, k + 2, k + 15, k + 16, k + 31, k + 32, k + 33, k + 66}:
        for at in {None, 0, 1, k - 2, k - 1, k, k + 1, 30, 31, 32, 33, 63, 64, length - 1}:
            if length < 1 or (at is not None and not 0 <= at < length):
                continue
            for what in ("n", "low"):
                start = int(rng.integers(0, 400 - length))
                r = genome[start:start + length].copy()
                q = np.full(length, 33 + 30, np.uint8)
                if at is not None and what == "n":
                    r[at] = ord("N")
                elif at is not None:
                    q[at] = 33 + 2
                reads.append(r)
                quals.append(q)
    bases, qual = np.concatenate(reads), np.concatenate(quals)
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    want = oracle.run(bases, qual, offsets, oracle.Params(k=k, min_count=1))
    rs = km.ReadSet(bases, qual, offsets)
    ka = km.KmerAnalysis(k, min_count=1, variant=variant)
    ka.submit(rs)
    assert_same(ka.results(), want, f"k={k} variant={variant}")
    ka.close()
    rs.close()
