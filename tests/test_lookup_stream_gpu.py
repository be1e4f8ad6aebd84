"""The first lookup of few k-mers among many survivors streams the survivors past them; the next one uses the index.
Both must give the survivors' own records: k-mers given twice, in either orientation, absent, and with bits above 2k."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)
MASK = (1 << 64) - 1


def words(values, W):
    return np.array([[(v >> (64 * (W - 1 - w))) & MASK for w in range(W)] for v in values], dtype=np.uint64)


def revcomp(v, k):
    r = 0
    for _ in range(k):
        r = (r << 2) | (3 - (v & 3))
        v >>= 2
    return r


@pytest.mark.parametrize("flags", [0, 4])
@pytest.mark.parametrize("k", [15, 31, 33, 77, 127])
def test_stream_and_index(k, flags):
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(k)
    n = 1_200_000
    genome = LETTERS[rng.integers(0, 4, n)]
    cut = list(range(0, n - k, 4000))
    reads = [genome[i:i + 4000 + k - 1] for i in cut]
    bases = np.concatenate(reads)
    offsets = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.uint64)
    rs = km.ReadSet(bases, np.full(len(bases), 33 + 40, np.uint8), offsets)
    ka = km.KmerAnalysis(k, min_count=1, flags=flags)
    ka.submit(rs)
    res = ka.results()
    assert len(res) >= 1 << 20
    W = res.keys.shape[1]
    pick = rng.integers(0, len(res), 3000)
    pick[100:200] = pick[:100]  # given twice
    vals = []
    for i in pick:
        v = 0
        for w in range(W):
            v = (v << 64) | int(res.keys[i, w])
        vals.append(v)
    turned = rng.random(len(vals)) < 0.5
    ask = [revcomp(v, k) if t else v for v, t in zip(vals, turned)]
    have = {tuple(r) for r in res.keys}
    absent = [int.from_bytes(rng.bytes(32), "big") & ((1 << (2 * k)) - 1) for _ in range(500)]
    beyond = [vals[0] | (1 << (2 * k))] if 2 * k % 64 else []
    q = words(ask + absent + beyond, W)
    first = ka.lookup(q)     # streams
    second = ka.lookup(q)    # builds the index
    third = ka.lookup(q[:7])
    assert np.array_equal(first, second) and np.array_equal(first[:7], third)
    m = len(ask)
    assert first["found"][:m].all()
    assert np.array_equal(first["flipped"][:m].astype(bool), turned)
    assert np.array_equal(first["count"][:m], res.count[pick])
    assert np.array_equal(first["ext"][:m], res.ext[pick])
    assert np.array_equal(first["cls"][:m], res.cls[pick])
    for i, v in enumerate(absent):
        assert bool(first["found"][m + i]) == (tuple(words([min(v, revcomp(v, k))], W)[0]) in have)
    assert not first["found"][m + len(absent):].any()
    ka.close()
    rs.close()
