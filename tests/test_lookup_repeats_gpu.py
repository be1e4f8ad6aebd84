"""K-mers given many times to the lookup that streams the survivors: one of them answers for all, in either
orientation, and a hundred thousand copies take no longer than as many different k-mers."""
import time

import numpy as np
import pytest

from tests.test_lookup_stream_gpu import LETTERS, revcomp, words

pytestmark = pytest.mark.gpu


def value(row):
    v = 0
    for w in row:
        v = (v << 64) | int(w)
    return v


@pytest.mark.parametrize("k", [31, 33, 77, 127])
def test_repeated_kmers(k):
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(k)
    n = 1_200_000
    genome = LETTERS[rng.integers(0, 4, n)]
    reads = [genome[i:i + 4000 + k - 1] for i in range(0, n - k, 4000)]
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    bases = np.concatenate(reads)
    rs = km.ReadSet(bases, np.full(len(bases), 33 + 40, np.uint8), offsets)
    ka = km.KmerAnalysis(k, min_count=1)
    ka.submit(rs)
    res = ka.results()
    W = res.keys.shape[1]
    m = 120_000  # below an eighth of the survivors: the first lookup streams them
    assert m <= len(res) // 8 and len(res) >= 1 << 20
    pick = rng.integers(0, len(res), m)
    distinct = res.keys[rng.permutation(len(res))[:m]]
    # 100 000 copies of one survivor in both orientations, 5 000 of an absent k-mer, the rest as drawn
    hot, absent = int(pick[0]), (1 << (2 * k)) - 1 - (0b01 << (k - 1))
    v = value(res.keys[hot])
    both = words([v, revcomp(v, k)], W)
    turned = rng.random(m) < 0.5
    q = res.keys[pick].copy()
    q[:100_000] = both[turned[:100_000].astype(int)]
    q[100_000:105_000] = words([absent], W)
    q[:] = q[(order := rng.permutation(m))]
    pick[:100_000] = hot
    want_found = np.ones(m, bool)
    want_found[100_000:105_000] = tuple(words([min(absent, revcomp(absent, k))], W)[0]) in {tuple(r) for r in res.keys}
    turned[100_000:] = False
    took = {}
    for name, keys in (("distinct", distinct), ("repeated", q)) * 2:  # the second time buffers are there
        ka.query()
        t = time.perf_counter()
        got = ka.lookup(keys)
        took[name] = time.perf_counter() - t
    second = ka.lookup(q)  # builds the index
    assert np.array_equal(got, second)
    want_found, turned, pick = want_found[order], turned[order], pick[order]
    assert np.array_equal(got["found"].astype(bool), want_found)
    assert np.array_equal(got["flipped"][want_found].astype(bool), turned[want_found])
    # query() runs again and the survivors' order is free: the records are compared through the index above and
    # with the first query's here
    assert np.array_equal(got["count"][want_found], res.count[pick][want_found])
    assert np.array_equal(got["ext"][want_found], res.ext[pick][want_found])
    assert np.array_equal(got["cls"][want_found], res.cls[pick][want_found])
    # the lookup of as many distinct k-mers takes about a millisecond; a slot for every copy would take 5e9 probes
    assert took["repeated"] < 10 * took["distinct"] + 5e-3, took
    ka.close()
    rs.close()
