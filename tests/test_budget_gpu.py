"""Queries of one handle while the device's free memory changes between them: one that is planned with an earlier
moment's free memory must not fail where a fresh plan fits, nor keep to waves and passes once the memory is back.
Each case runs in a process of its own, so that nothing else holds device memory."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SETUP = """
import ctypes
import numpy as np
import torch
import paper_1809_07014_gb300 as km

LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)
N, L, K = 1_200_000, 80, 31
rng = np.random.default_rng(1)


def leave(free):
    # takes all device memory but `free` bytes (the library's pool gives its unused memory back first)
    cu = ctypes.CDLL("libcuda.so.1")
    pool, dev = ctypes.c_void_p(), ctypes.c_int()
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    assert cu.cuMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    torch.cuda.synchronize()
    return torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")


def readset(reads):
    bases = np.ascontiguousarray(reads).reshape(-1)
    offsets = np.arange(len(reads) + 1, dtype=np.uint64) * np.uint64(L)
    return km.ReadSet(bases, np.full(len(bases), 73, np.uint8), offsets)


def pairs():
    # every read twice, a thousand of them three times
    half = LETTERS[rng.integers(0, 4, (N // 2, L))]
    reads = np.concatenate([half, half])
    reads[-1000:] = half[:1000]
    return readset(reads)


def same(a, b):
    return a.windows == b.windows and all(np.array_equal(getattr(a, c), getattr(b, c))
                                          for c in ("keys", "count", "ext", "cls"))


torch.zeros(1, device="cuda")
"""

# the gate makes the first query small (no k-mer twice) and the second large (every k-mer twice)
TAKEN = SETUP + """
P = dict(min_count=3, flags=km.KMER_FLAG_BLOOM_GATE | km.KMER_FLAG_SORTED_OUTPUT)
single, double = readset(LETTERS[rng.integers(0, 4, (N, L))]), pairs()
ref = km.KmerAnalysis(K, **P)
ref.submit(double)
want = ref.results()
assert len(want) >= 50_000 - 100, len(want)
ref.close()
ka = km.KmerAnalysis(K, **P)
ka.submit(single)
ka.query()
ka.reset()
hog = leave(900 << 20)
ka.submit(double)
got = ka.results()
st = ka.stats()
assert same(got, want)
assert st["passes"] > 1 or st["l2_waves"] > 0, st
"""

FREED = SETUP + """
rs = pairs()
ka = km.KmerAnalysis(K, min_count=3, flags=km.KMER_FLAG_SORTED_OUTPUT)
hog = leave(1500 << 20)
ka.submit(rs)
tight = ka.results()
st = ka.stats()
assert st["passes"] > 1 or st["l2_waves"] > 0, st
del hog
torch.cuda.empty_cache()
wide = ka.results(ka.query())
st = ka.stats()
assert st["passes"] == 1 and st["l2_waves"] == 0, st
assert same(wide, tight)
"""


@pytest.mark.parametrize("name", ["TAKEN", "FREED"])
def test_free_memory_changes_between_queries(name):
    r = subprocess.run([sys.executable, "-c", globals()[name]], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
