"""Contigs in host memory that the merge cuts into pieces: the same set as from device memory (offsets that do not start
at 0 included), and no copy of every contig on the host, which takes three times as long as the rest."""
import time

import numpy as np
import pytest

from tests.test_lookup_stream_gpu import LETTERS

pytestmark = pytest.mark.gpu


def handle(k, rng):
    import paper_1809_07014_gb300 as km
    reads = LETTERS[rng.integers(0, 4, (4000, 150))]
    rs = km.ReadSet(reads.reshape(-1), np.full(reads.size, 73, np.uint8), np.arange(4001, dtype=np.uint64) * 150)
    ka = km.KmerAnalysis(k, flags=km.KMER_FLAG_SORTED_OUTPUT)
    ka.submit(rs)
    return ka, rs


# pieces hold max(256, 4 (k + 1)) bases
@pytest.mark.parametrize("k", [21, 33, 77, 127])
def test_host_and_device_contigs(k):
    import torch
    rng = np.random.default_rng(k)
    ka, rs = handle(k, rng)
    lengths = [0, k - 1, k, 255, 256, 257, 511, 512, 513, 1025, 40_000] + list(rng.integers(1, 2000, 300))
    for first in (0, 777):
        offs = (first + np.concatenate([[0], np.cumsum(lengths)])).astype(np.uint64)
        seq = LETTERS[rng.integers(0, 4, int(offs[-1]))]
        seq[rng.integers(first, len(seq), 200)] = ord("N")
        ka.query()
        host = ka.merge_contigs(seq, offs)
        launches = ka.stats()["launches"]
        ka.query()
        dev = ka.merge_contigs(torch.from_numpy(seq).cuda(), torch.from_numpy(offs.view(np.int64)).cuda())
        assert ka.stats()["launches"] == launches  # cut on the device both times
        for c in ("keys", "count", "ext", "cls"):
            np.testing.assert_array_equal(getattr(host, c), getattr(dev, c))
    bad = offs.copy()
    bad[5] = bad[3] - np.uint64(1)
    ka.query()
    import paper_1809_07014_gb300 as km
    with pytest.raises(km.KmerError) as e:
        ka.merge_contigs(seq, bad)
    assert e.value.code == km.KMER_ERR_INVALID_ARG
    ka.close()
    rs.close()


def test_host_contigs_take_no_longer_for_being_cut():
    import paper_1809_07014_gb300 as km
    rng = np.random.default_rng(0)
    ka, rs = handle(31, rng)
    took = {}
    for length in (250, 600):
        n = 60_000_000 // length
        seq = LETTERS[rng.integers(0, 4, n * length)]
        offs = np.arange(n + 1, dtype=np.uint64) * np.uint64(length)
        for _ in range(4):
            ka.query()
            t = time.perf_counter()
            km.kmer_analysis_merge_contigs(ka.handle, seq.ctypes.data, offs.ctypes.data, n, km.KMER_HOST)
            took[length] = min(took.get(length, 1e9), time.perf_counter() - t)
    assert took[600] < 2 * took[250], took
    ka.close()
    rs.close()
