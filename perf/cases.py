"""Workloads of the k-mer analysis library, timed through its public entry points.

The inputs are synthetic reads of the shapes that the package's benchmark and
tests use: genomes of random bases mixed with log-normal abundance, reads from
both strands, substitutions whose bases have low Phred qualities, a few Ns, or
one small genome read 30 times.  They are drawn on the GPU from the seed.

The k-mer set is a set: without ``KMER_FLAG_SORTED_OUTPUT`` its order differs
from run to run.  A program that keeps or compares results asks for ascending
key order, as most cases here do; one that only consults the table looks
k-mers up, as the "markers" cases do after the default, unordered query.
"""
import math

import torch

import paper_1809_07014_gb300 as km

# One sample of reads: `reads` of len_lo..len_hi bases from `genomes` genomes of glen_lo..glen_hi bases, abundance
# LogNormal(0, sigma), substitution rate `err`; `low`: substituted bases get Phred 2..12 and one base in 10^4 is N.
_META = {"genomes": 50, "glen_lo": 1_000_000, "glen_hi": 5_000_000, "sigma": 1.5, "err": 0.01, "low": True,
         "len_lo": 150, "len_hi": 150}
_SINGLE = {"genomes": 1, "glen_lo": 100_000, "glen_hi": 100_000, "sigma": 0.0, "err": 0.005, "low": False,
           "len_lo": 150, "len_hi": 150}
_LADDER = (21, 33, 55, 77, 99)   # the k of one iterative assembly
_MIXED = (21, 33, 55)            # the k of a collection of samples


def listed():
    return [
        # a handful of reads of one small genome (an amplicon, a plasmid, a test): launches and latency count
        dict(_SINGLE, name="small_k21", mode="count", k=21, reads=2_000),
        # one assembly's ladder of k over one resident read set: five short analyses, one to four key words
        dict(_SINGLE, name="ladder_20k_reads", mode="ladder", reads=20_000),
        # a small metagenome sample, two key words
        dict(_META, name="sample_50M_k55", mode="count", k=55, genomes=20, reads=333_333),
        # trimmed reads of uneven lengths, three key words, the static extension rule and a higher count threshold
        dict(_META, name="trimmed_100M_k77", mode="count", k=77, genomes=25, reads=613_497, len_lo=75, len_hi=251,
             min_count=3, ext_mode=1),
        # the last, longest k of an assembly, four key words
        dict(_META, name="sample_300M_k99", mode="count", k=99, genomes=50, reads=2_000_001),
        # a sequencing run as a whole, the default k, in key order
        dict(_META, name="run_1G_k31", mode="count", k=31, reads=6_666_667),
        # the headline workload in the default, unordered form; then the marker k-mers of one genome are looked up
        dict(_META, name="run_2G_k31_markers", mode="markers", k=31, reads=13_333_334, markers=1_000_003),
        # memory is tight and most k-mers are seen once: the Bloom gate before counting
        dict(_META, name="gated_300M_k55", mode="gated", k=55, genomes=50, reads=2_000_000),
        # one iteration of the assembly: k-mers, contigs, the next k's k-mers, merged with the contigs' k-mers
        dict(_META, name="iteration_200M_k31", mode="iteration", k=31, next_k=41, genomes=10, reads=1_333_333),
        # a collection of samples of uneven size and mixed k, run as one batch
        dict(_META, name="batch_8", mode="batch", genomes=10, reads=40_000, reads_hi=666_667, jobs=8, min_count=3),
        # requests of mixed size and k served by four workers at once, results handed over in host memory
        dict(_META, name="serve_6", mode="serve", genomes=10, reads=6_667, reads_hi=66_667, jobs=6),
        # reads and results in page-locked host memory, as a sequencing pipeline hands them over
        dict(_META, name="host_20M_k33", mode="host", k=33, genomes=10, reads=133_331),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mode = rng.choice(("count", "count", "count", "count", "markers", "ladder", "gated", "iteration", "batch", "serve",
                       "host"))
    c = dict(_META, mode=mode, genomes=rng.randint(10, 50))
    if rng.random() < 0.3:  # uneven read lengths
        c["len_lo"] = rng.randint(50, 150)
        c["len_hi"] = rng.randint(151, 301)
    mean_len = (c["len_lo"] + c["len_hi"]) / 2

    def reads(lo_bases, hi_bases):
        return max(1, int(_log_int(rng, lo_bases, hi_bases) / mean_len))

    if mode == "count":
        c["k"] = rng.choice((21, 25, 31, 31, 33, 41, 55, 63, 77, 99))
        if rng.random() < 0.25:
            c.update(_SINGLE, glen_lo=rng.randint(20_000, 200_000))
            c["glen_hi"] = c["glen_lo"]
            c["reads"] = rng.randint(1_000, 40_000)
        else:
            c["reads"] = reads(1e6, 1e9 * 32 / (c["k"] + 1))
        c["min_count"] = rng.choice((2, 2, 2, 3))
        c["ext_mode"] = rng.choice((0, 0, 1))
    elif mode == "markers":
        c.update(k=rng.choice((21, 31, 55)), reads=reads(5e6, 1e9), markers=_log_int(rng, 1_000, 4_000_000))
    elif mode == "ladder":
        c.update(_SINGLE, glen_lo=rng.randint(50_000, 200_000), reads=rng.randint(5_000, 60_000))
        c["glen_hi"] = c["glen_lo"]
    elif mode == "gated":
        c.update(k=rng.choice((31, 33, 55)), reads=reads(2e7, 5e8))
    elif mode == "iteration":
        k = rng.choice((21, 31, 41))
        c.update(k=k, next_k=k + rng.choice((2, 10, 20)), genomes=rng.randint(5, 20), reads=reads(2e7, 3e8))
    elif mode == "batch":
        c["reads"] = reads(5e6, 2e7)
        c["reads_hi"] = c["reads"] * rng.randint(2, 6)
        c["jobs"] = rng.randint(4, 10)
        c["min_count"] = rng.choice((3, 4))
    elif mode == "serve":
        c["reads"] = reads(1e6, 3e6)
        c["reads_hi"] = c["reads"] * rng.randint(2, 6)
        c["jobs"] = rng.randint(3, 8)
    else:
        c.update(k=rng.choice((21, 31, 33, 55)), reads=reads(2e6, 3e7))
    return c


# ------------------------------------------------------------------ inputs
def _genomes(case, gen):
    lens = torch.randint(case["glen_lo"], case["glen_hi"] + 1, (case["genomes"],), generator=gen, device="cuda")
    starts = torch.cumsum(lens, 0) - lens
    codes = torch.randint(0, 4, (int(lens.sum()),), generator=gen, device="cuda", dtype=torch.uint8)
    return codes, lens, starts


def _sample(case, n_reads, gen, genomes=None):
    """Reads of one sample: (bases, quals, offsets) on the GPU."""
    codes, lens, starts = genomes if genomes is not None else _genomes(case, gen)
    dev = "cuda"
    weight = lens.double() * torch.exp(case["sigma"] * torch.randn(len(lens), generator=gen, device=dev,
                                                                   dtype=torch.float64))
    edges = torch.cumsum(weight, 0)
    lo, hi = case["len_lo"], case["len_hi"]
    rlen = torch.randint(lo, hi + 1, (n_reads,), generator=gen, device=dev)
    offsets = torch.zeros(n_reads + 1, dtype=torch.int64, device=dev)
    torch.cumsum(rlen, 0, out=offsets[1:])
    total = n_reads * lo if lo == hi else int(offsets[-1])
    bases = torch.empty(total, dtype=torch.uint8, device=dev)
    quals = torch.empty(total, dtype=torch.uint8, device=dev)
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)
    col = torch.arange(hi, device=dev)
    step = max(1, 150_000_000 // hi)
    at = 0
    for r0 in range(0, n_reads, step):
        n = min(step, n_reads - r0)
        L = rlen[r0:r0 + n]
        pick = torch.rand(n, generator=gen, device=dev, dtype=torch.float64) * edges[-1]
        g = torch.searchsorted(edges, pick).clamp_(max=len(lens) - 1)
        p = starts[g] + (torch.rand(n, generator=gen, device=dev, dtype=torch.float64) * (lens[g] - L + 1)).long()
        rev = torch.rand(n, generator=gen, device=dev) < 0.5
        first = torch.where(rev, p + L - 1, p)
        sign = torch.where(rev, -1, 1)
        idx = first[:, None] + sign[:, None] * col[None, :]
        c = codes[idx.clamp_(0, len(codes) - 1)]
        del idx
        c ^= torch.where(rev, 3, 0).to(torch.uint8)[:, None]
        q = torch.randn((n, hi), generator=gen, device=dev).mul_(5).add_(32).round_().clamp_(2, 41).to(torch.uint8)
        bad = torch.rand((n, hi), generator=gen, device=dev) < case["err"]
        c = torch.where(bad, (c + torch.randint(1, 4, (n, hi), generator=gen, device=dev, dtype=torch.uint8)) & 3, c)
        b = letters[c.long()]
        if case["low"]:
            q = torch.where(bad, torch.randint(2, 13, (n, hi), generator=gen, device=dev, dtype=torch.uint8), q)
            un = torch.rand((n, hi), generator=gen, device=dev) < 1e-4
            b = torch.where(un, 78, b)
            q = torch.where(un, 2, q)
        q += 33
        if lo != hi:
            keep = col[None, :] < L[:, None]
            b, q = b[keep], q[keep]
        bases[at:at + b.numel()] = b.reshape(-1)
        quals[at:at + q.numel()] = q.reshape(-1)
        at += b.numel()
    return bases, quals, offsets


def _sizes(case):
    """Reads of each job of a batch or a request mix, log-spaced from `reads` to `reads_hi`."""
    n = case["jobs"]
    return [int(round(case["reads"] * (case["reads_hi"] / case["reads"]) ** (i / max(1, n - 1)))) for i in range(n)]


def _params(case):
    return {"min_count": case.get("min_count", 2), "ext_mode": case.get("ext_mode", 0),
            "flags": km.KMER_FLAG_SORTED_OUTPUT}


def _words(k):
    return (2 * k + 63) // 64


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _arrays(case, n_reads, k, pin=False):
    """The program's own result arrays.  At most 30 in 100 windows of randomly placed reads give a survivor (P(depth >= 2) /
    depth of a Poisson depth is below 0.3 everywhere); rows past the last survivor stay zero."""
    cap = 3 * n_reads * case["len_hi"] // 10 + 1024
    where = {"pin_memory": True} if pin else {"device": "cuda"}
    return (torch.zeros((cap, _words(k)), dtype=torch.int64, **where), torch.zeros(cap, dtype=torch.int32, **where),
            torch.zeros((cap, 8), dtype=torch.int32, **where), torch.zeros((cap, 2), dtype=torch.uint8, **where))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    mode = case["mode"]
    st = {"case": case}
    if mode in ("batch", "serve"):
        genomes = _genomes(case, gen)
        st["sets"] = [km.ReadSet(*_sample(case, n, gen, genomes)) for n in _sizes(case)]
        ks = [(_MIXED if mode == "batch" else _LADDER)[i % (3 if mode == "batch" else 5)] for i in range(case["jobs"])]
        st["outs"] = [_arrays(case, n, k, pin=mode == "serve") for n, k in zip(_sizes(case), ks)]
        if mode == "batch":
            st["batch"] = km.Batch([(rs, {"k": k, "min_count": case["min_count"]}) for rs, k in zip(st["sets"], ks)])
        else:
            st["server"] = km.Server(workers=4)
        st["ks"] = ks
        return st
    genomes = _genomes(case, gen)
    reads = _sample(case, case["reads"], gen, genomes)
    if mode == "ladder":
        st["set"] = km.ReadSet(*reads)
        st["jobs"] = []
        for k in _LADDER:
            ka = km.KmerAnalysis(k, **_params(case))
            ka.submit(st["set"])
            st["jobs"].append((ka, _arrays(case, case["reads"], k)))
        return st
    if mode == "host":
        reads = tuple(_pinned(t) for t in reads)
    st["reads"] = reads
    st["set"] = km.ReadSet(*reads)
    p = _params(case)
    if mode == "markers":
        p["flags"] = 0
        st["keys"] = _markers(case, genomes[0], gen)
        st["records"] = torch.zeros((case["markers"], km.KMER_RECORD_DTYPE.itemsize), dtype=torch.uint8, device="cuda")
    else:
        st["out"] = _arrays(case, case["reads"], case.get("next_k", case["k"]), pin=mode == "host")
    if mode == "gated":
        p["flags"] |= km.KMER_FLAG_BLOOM_GATE
    st["ka"] = km.KmerAnalysis(case["k"], **p)
    if mode == "iteration":
        st["next"] = km.KmerAnalysis(case["next_k"], **p)
        st["contigs"] = (torch.zeros(3 * case["reads"] * case["len_hi"] // 10, dtype=torch.uint8, device="cuda"),
                         torch.zeros(case["reads"], dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()
    return st


def _markers(case, codes, gen):
    """k-mers at random places of the genomes, one in eight with a base changed (mostly absent from the reads)."""
    k, n, W = case["k"], case["markers"], _words(case["k"])
    p = torch.randint(0, len(codes) - k + 1, (n,), generator=gen, device="cuda")
    change = torch.randint(0, 8 * k, (n,), generator=gen, device="cuda")
    words = torch.zeros((n, W), dtype=torch.int64, device="cuda")
    for j in range(k):
        bit = 2 * (k - 1 - j)
        w = W - 1 - bit // 64
        c = codes[p + j].long() ^ (change == j).long()
        words[:, w] |= c << (bit % 64)
    return words


# --------------------------------------------------------------------- run
class _Device:
    """Device memory owned by a library object, as an array (keeps the object alive)."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (int(ptr), False), "shape": shape, "typestr": typestr, "version": 3}


def _tensor(owner, ptr, shape, typestr, dtype):
    if not ptr or 0 in shape:
        return torch.empty(shape, dtype=dtype, device="cuda")
    return torch.as_tensor(_Device(owner, ptr, shape, typestr), device="cuda")


def _view(owner, v):
    n, W = int(v.n), int(v.words)
    return (_tensor(owner, v.keys, (n, W), "<i8", torch.int64), _tensor(owner, v.count, (n,), "<i4", torch.int32),
            _tensor(owner, v.ext, (n, 8), "<i4", torch.int32), _tensor(owner, v.cls, (n, 2), "|u1", torch.uint8))


def _result(out, v, distinct=True):
    r = dict(zip(("keys", "count", "ext", "cls"), out), n=int(v.n), windows=int(v.windows))
    if distinct:  # a gate's number of distinct k-mers includes its false positives, which differ from run to run
        r["distinct"] = int(v.distinct)
    return r


def _analyse(st, ka):
    """Count the read set; the survivors stay in the analysis's own device memory."""
    ka.reset()
    ka.submit(st["set"])
    return ka.query()


def _query_into(ka, out, where):
    return km.kmer_analysis_query_into(ka.handle, *(t.data_ptr() for t in out), len(out[1]), where)


def run(st):
    mode = st["case"]["mode"]
    if mode == "ladder":
        return [_result(out, _query_into(ka, out, km.KMER_DEVICE)) for ka, out in st["jobs"]]
    if mode == "batch":
        return _run_batch(st)
    if mode == "serve":
        return _run_server(st)
    ka = st["ka"]
    st["set"].pack(*st["reads"])
    if mode == "markers":
        v = _analyse(st, ka)
        km.kmer_analysis_lookup(ka.handle, st["keys"].data_ptr(), len(st["keys"]), st["records"].data_ptr(),
                                km.KMER_DEVICE)
        return {"records": st["records"], "n": int(v.n), "windows": int(v.windows), "distinct": int(v.distinct)}
    if mode == "iteration":
        return _run_iteration(st)
    ka.reset()
    ka.submit(st["set"])
    v = _query_into(ka, st["out"], km.KMER_HOST if mode == "host" else km.KMER_DEVICE)
    return _result(st["out"], v, distinct=mode != "gated")


def _run_iteration(st):
    ka, nxt = st["ka"], st["next"]
    _analyse(st, ka)
    c = km.kmer_analysis_traverse(ka.handle)
    nc = int(c.n_contigs)
    seq, offs = st["contigs"]
    km.kmer_analysis_copy_contigs(ka.handle, seq.data_ptr(), offs.data_ptr(), len(seq), len(offs) - 1)
    _analyse(st, nxt)
    added, v = km.kmer_analysis_merge_contigs(nxt.handle, seq.data_ptr(), offs.data_ptr(), nc, km.KMER_DEVICE)
    for to, t in zip(st["out"], _view(nxt, v)):
        to[:len(t)].copy_(t)
    return dict(_result(st["out"], v), contigs=seq, contig_offsets=offs, n_contigs=nc, added=int(added))


def _run_batch(st):
    # a batch leaves each sample's k-mers unordered; the program puts them in a fixed order (of a mix of the key words)
    b = st["batch"]
    b.run()
    res = []
    for i, out in enumerate(st["outs"]):
        v = b.view(i)
        got = _view(b, v)
        mix = got[0][:, -1] if got[0].shape[1] == 1 else got[0][:, 0] * 0x3C6EF372FE94F82B + got[0][:, 1]
        order = torch.argsort(mix)
        for to, t in zip(out, got):
            if t.dim() > 1:  # eight bytes, or both class bytes, at a time
                wide = torch.int16 if t.dtype == torch.uint8 else torch.int64
                for j in range(t.view(wide).shape[1]):
                    to.view(wide)[:len(t), j] = t.view(wide)[:, j][order]
            else:
                to[:len(t)] = t[order]
        res.append(_result(out, v))
    return res


def _run_server(st):
    srv = st["server"]
    ids = [srv.submit(rs, k, flags=km.KMER_FLAG_SORTED_OUTPUT) for rs, k in zip(st["sets"], st["ks"])]
    res = []
    for i, out in zip(ids, st["outs"]):
        v, _ = srv.wait(i)
        km.kmer_server_copy_results(srv.handle, i, *(t.data_ptr() for t in out), len(out[1]))
        res.append(_result(out, v))
    for i in ids:
        srv.release(i)
    return res


# -------------------------------------------------------------------- work
def _expected_survivors(case, n_reads, k):
    """Genome positions whose k-mer is read correctly at least twice (Poisson depth, log-normal abundance)."""
    L = (case["len_lo"] + case["len_hi"]) / 2
    windows = n_reads * max(0.0, L - k + 1)
    size = case["genomes"] * (case["glen_lo"] + case["glen_hi"]) / 2
    s = case["sigma"]
    need = case.get("min_count", 2)
    hit = 0.0
    for i in range(64):  # the middle of each of 64 slices of [-4, 4] standard deviations
        x = -4 + 8 * (i + 0.5) / 64
        share = math.exp(-x * x / 2) / math.sqrt(2 * math.pi) * 8 / 64
        lam = windows / size * math.exp(s * x - s * s / 2) * (1 - case["err"]) ** k
        p = term = math.exp(-lam)
        for j in range(1, need):
            term *= lam / j
            p += term
        hit += share * (1 - p)
    return size * hit


def work(case):
    """The reads (a base and a quality byte per base, an offset per read) read once, the survivors written once."""
    mean_len = (case["len_lo"] + case["len_hi"]) / 2

    def one(n_reads, k, packed=False):
        # 2 bytes a base; reads that are already resident and packed: half a byte a base
        return n_reads * (mean_len * (0.5 if packed else 2.0) + 8) + _expected_survivors(case, n_reads, k) * (8 * _words(k) + 38)

    mode = case["mode"]
    if mode == "ladder":
        total = sum(one(case["reads"], k, True) for k in _LADDER)
    elif mode in ("batch", "serve"):
        ks = _MIXED if mode == "batch" else _LADDER
        total = sum(one(n, ks[i % len(ks)], True) for i, n in enumerate(_sizes(case)))
    elif mode == "markers":
        L = case["reads"] * (mean_len * 2 + 8)
        total = L + case["markers"] * (8 * _words(case["k"]) + 40)
    elif mode == "iteration":  # the reads once, the second k-mer set and the contigs written
        n = _expected_survivors(case, case["reads"], case["k"])
        total = one(case["reads"], case["next_k"]) + n
    else:
        total = one(case["reads"], case["k"])
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """Every output is a whole number (keys, counts, tallies, classes, bases), so there is nothing to round."""
    return None
