"""Packing at its edges: reads of 0 to 97 bases that begin at every byte alignment of the device buffer, its first and
last bytes included, every byte value as a base, and qualities on both sides of the threshold.  Compared with the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 4, 7, 8, 13, 15])
@pytest.mark.parametrize("offset,threshold", [(0, 0), (33, 20), (64, 63), (64, 64), (100, 155), (100, 156)])
def test_edges(shift, offset, threshold):
    import torch
    import oracle
    import paper_1809_07014_gb300 as km
    from tests.helpers import assert_same

    rng = np.random.default_rng(threshold * 16 + shift)
    lengths = np.concatenate([rng.integers(0, 98, 300), [0, 1, 31, 32, 33, 63, 64, 65, 0, 5 + shift]])
    offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.uint64)
    n = int(offsets[-1])
    bases = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n)]
    odd = rng.random(n) < 0.01
    bases[odd] = rng.integers(0, 256, int(odd.sum()))
    near = np.clip(offset + threshold + rng.integers(-1, 2, n), 0, 255)
    quals = np.where(rng.random(n) < 0.5, near, rng.integers(0, 256, n)).astype(np.uint8)

    want = oracle.run(bases, quals, offsets,
                      oracle.Params(k=5, min_count=1, qual_offset=offset, qual_threshold=threshold))
    # the arrays end where their buffers end
    dev = [torch.from_numpy(np.concatenate([np.full(shift, 65, np.uint8), a])).cuda()[shift:] for a in (bases, quals)]
    rs = km.ReadSet(dev[0], dev[1], torch.from_numpy(offsets.view(np.int64)).cuda(), qual_offset=offset,
                    qual_threshold=threshold)
    ka = km.KmerAnalysis(5, min_count=1, qual_offset=offset, qual_threshold=threshold)
    ka.submit(rs)
    assert_same(ka.results(), want, f"shift={shift} quality {offset}+{threshold}")
    ka.close()
    rs.close()
