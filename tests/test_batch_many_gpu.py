"""Batches of many small deep samples: a job brings its share of the leaves that fill the GPU, not all of them.  Results
equal separate analyses; the time stays near that of the same batch with as few leaves as its k-mers need."""
import time

import numpy as np
import pytest

from tests.test_lookup_stream_gpu import LETTERS

pytestmark = pytest.mark.gpu


def sample(rng, reads, genome):
    import paper_1809_07014_gb300 as km
    g = rng.integers(0, 4, genome, dtype=np.uint8)
    bases = LETTERS[g[rng.integers(0, genome - 150, reads)[:, None] + np.arange(150)]].reshape(-1)
    return km.ReadSet(bases, np.full(len(bases), 73, np.uint8), np.arange(reads + 1, dtype=np.uint64) * np.uint64(150))


def in_order(r):
    o = np.lexsort([r.keys[:, w] for w in reversed(range(r.keys.shape[1]))])
    return r.windows, r.distinct, r.keys[o], r.count[o], r.ext[o], r.cls[o]


# one large job among small ones, jobs of every key width, one job alone, an empty one
@pytest.mark.parametrize("shapes", [[(60_000, 200_000, 31)] + [(300, 2000, 31)] * 20,
                                    [(1300, 10_000, k) for k in (21, 31, 33, 55, 77, 99, 127)] * 3,
                                    [(1300, 10_000, 31)], [(1300, 10_000, 55), (0, 1000, 55)]])
def test_same_as_separate_analyses(shapes):
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(len(shapes))
    sets = [sample(rng, n, g) for n, g, _ in shapes]
    b = km.Batch([(s, {"k": k}) for s, (_, _, k) in zip(sets, shapes)])
    for _ in range(3):  # the second and third runs are planned from the first one's counts
        b.run()
        for i, (s, (_, _, k)) in enumerate(zip(sets, shapes)):
            ka = km.KmerAnalysis(k)
            ka.submit(s)
            for x, y in zip(in_order(b.results(i)), in_order(ka.results())):
                np.testing.assert_array_equal(x, y)
            ka.close()
    b.close()
    for s in sets:
        s.close()


def test_many_small_jobs_take_few_leaves_each():
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(0)
    sets = [sample(rng, 1300, 10_000) for _ in range(300)]
    took = {}
    for name, extra in (("few", {"leaf_bits": 3}), ("own", {})):
        b = km.Batch([(s, {"k": 31, "distinct_hint": 10_000, **extra}) for s in sets])
        for _ in range(6):
            t = time.perf_counter()
            b.run()
            took[name] = min(took.get(name, 1e9), time.perf_counter() - t)
        b.close()
    for s in sets:
        s.close()
    assert took["own"] < 1.4 * took["few"], took  # 256 leaves each: 2.1 times
