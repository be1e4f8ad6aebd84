// Point lookups of k-mers among the survivors of a query: the read side of
// the k-mer table that the later stages of Algorithm 1 consult (the de
// Bruijn graph walks of Sec. II-C ask, for a k-mer, its count and the class
// of each side).  An index over the compacted survivors -- an open-addressing
// table of survivor positions in HBM -- is built once per query; each lookup
// canonicalises the given k-mer (Sec. II-B: a k-mer and its reverse
// complement are one vertex) and probes the index.
#include "kernels.h"
#include "keyops.cuh"
#include "kmer_analysis.h"

namespace kmer {

template <int W>
__global__ void __launch_bounds__(256) index_build_kernel(const unsigned long long* __restrict__ keys,
                                                          unsigned long long n, unsigned k,
                                                          unsigned* __restrict__ idx, unsigned long long cap) {
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * 256) {
        unsigned long long key[W];
#pragma unroll
        for (int w = 0; w < W; ++w) key[w] = keys[i * W + w];
        unsigned long long s = index_home<W>(key, k, cap);
        // survivors are distinct keys: the first empty slot of the sequence is ours
        for (unsigned long long probe = 0; probe < cap; ++probe) {
            if (atomicCAS(idx + s, kIdxEmpty, (unsigned)i) == kIdxEmpty) break;
            s = (s + 1) & (cap - 1);
        }
    }
}

template <int W>
__global__ void __launch_bounds__(256) lookup_kernel(const unsigned long long* __restrict__ q, unsigned long long n,
                                                     const unsigned k, const unsigned* __restrict__ idx,
                                                     unsigned long long cap, const unsigned long long* __restrict__ keys,
                                                     const unsigned* __restrict__ count,
                                                     const unsigned* __restrict__ ext,
                                                     const unsigned char* __restrict__ cls,
                                                     kmer_record* __restrict__ out) {
    const unsigned hb = 2 * k - 64 * (W - 1);
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * 256) {
        unsigned long long key[W], rc[W];
#pragma unroll
        for (int w = 0; w < W; ++w) key[w] = q[i * W + w];
        kmer_record r{};
        const bool valid = hb >= 64 || (key[0] >> hb) == 0ull;  // no bits above 2k
        if (valid) {
            reverse_complement<W>(key, k, rc);
            bool flip = false;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (key[w] != rc[w]) {
                    flip = rc[w] < key[w];
                    break;
                }
            }
            if (flip) {
#pragma unroll
                for (int w = 0; w < W; ++w) key[w] = rc[w];
            }
            r.flipped = flip ? 1 : 0;
            unsigned long long s = index_home<W>(key, k, cap);
            for (unsigned long long probe = 0; probe < cap; ++probe) {
                const unsigned p = idx[s];
                if (p == kIdxEmpty) break;
                bool same = true;
#pragma unroll
                for (int w = 0; w < W; ++w) same = same && keys[(unsigned long long)p * W + w] == key[w];
                if (same) {
                    r.found = 1;
                    r.count = count[p];
#pragma unroll
                    for (int e = 0; e < 8; ++e) r.ext[e] = ext[(unsigned long long)p * 8 + e];
                    r.cls[0] = cls[2ull * p];
                    r.cls[1] = cls[2ull * p + 1];
                    break;
                }
                s = (s + 1) & (cap - 1);
            }
        }
        out[i] = r;
    }
}

// The other way round: a few k-mers looked up once among many survivors need
// no index of the survivors.  The k-mers go into a table of their own (eight
// bytes a slot: 32 bits of z's mix, number + 1), in the order of z, and all
// survivors stream past it once: the partitions come out in that order too, so
// the slots a survivor needs are in L1 or L2.  1 M k-mers among 101 M
// survivors: 0.77 ms, against 4.0 for the index.
//
// A k-mer given many times (in either orientation) takes one slot: the copy
// that claims it answers for the others, rep[i] names it, and a last pass
// hands its record on.  With a slot for every copy, m copies would probe past
// each other m^2 / 2 times and leave one run of m slots in the way of every
// survivor that starts in it.  Among 101 M survivors, 1 M different k-mers, all
// of them found: 0.98 ms (0.97 without this); 1 M copies of one: 0.32 ms (0.90
// if every copy tried the compare-and-swap before it read the slot).

// The canonical form of a given k-mer; returns whether it is the reverse complement.
template <int W>
__device__ __forceinline__ bool canonical_of(const unsigned long long* __restrict__ q, unsigned long long i, unsigned k,
                                             unsigned long long (&key)[W]) {
    unsigned long long rc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) key[w] = q[i * W + w];
    reverse_complement<W>(key, k, rc);
    const bool flip = key_less<W>(rc, key);
#pragma unroll
    for (int w = 0; w < W; ++w) key[w] = flip ? rc[w] : key[w];
    return flip;
}

template <int W>
__global__ void __launch_bounds__(256) wanted_build_kernel(const unsigned long long* __restrict__ q,
                                                           unsigned long long n, const unsigned k,
                                                           unsigned long long* __restrict__ canon,
                                                           unsigned long long* table, unsigned long long cap,
                                                           unsigned* __restrict__ rep, kmer_record* __restrict__ out) {
    const unsigned hb = 2 * k - 64 * (W - 1), sh = __clzll((long long)cap) + 1;
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * 256) {
        kmer_record r{};
        unsigned mine = (unsigned)i;
        if (q[i * W] >> hb == 0ull) {  // no bits above 2k (hb is below 64 for odd k)
            unsigned long long key[W];
            r.flipped = canonical_of<W>(q, i, k, key) ? 1 : 0;
#pragma unroll
            for (int w = 0; w < W; ++w) canon[i * W + w] = key[w];
            const unsigned long long z = aligned_z<W>(key, k);
            const unsigned long long word = (mix_z(z) >> 32) << 32 | (unsigned)(i + 1);
            unsigned long long s = z >> sh;
            // slots fill and never empty, so copies of a k-mer meet in the first
            // slot of its sequence that any of them claims
            for (unsigned long long probe = 0; probe < cap; ++probe) {
                unsigned long long e = *(volatile unsigned long long*)(table + s);
                if (e == 0ull) e = atomicCAS(table + s, 0ull, word);
                if (e == 0ull) break;  // claimed
                if ((e ^ word) >> 32 == 0ull) {
                    unsigned long long other[W];
                    const unsigned j = (unsigned)e - 1u;
                    canonical_of<W>(q, j, k, other);
                    bool same = true;
#pragma unroll
                    for (int w = 0; w < W; ++w) same = same && other[w] == key[w];
                    if (same) {
                        mine = j;
                        break;
                    }
                }
                s = (s + 1) & (cap - 1);
            }
        }
        rep[i] = mine;
        out[i] = r;  // not found, until a survivor says otherwise
    }
}

template <int W>
__global__ void __launch_bounds__(256) wanted_stream_kernel(const unsigned long long* __restrict__ keys,
                                                            unsigned long long n, const unsigned k,
                                                            const unsigned long long* __restrict__ canon,
                                                            const unsigned long long* __restrict__ table,
                                                            unsigned long long cap, const unsigned* __restrict__ count,
                                                            const unsigned* __restrict__ ext,
                                                            const unsigned char* __restrict__ cls,
                                                            kmer_record* __restrict__ out) {
    constexpr int U = 4;  // survivors per thread and step: their slots are read together
    const unsigned sh = __clzll((long long)cap) + 1;
    const unsigned lane = threadIdx.x & 31u;
    for (unsigned long long i0 = (blockIdx.x * 256ull + (threadIdx.x & ~31u)) * U + lane; i0 < n;
         i0 += (unsigned long long)gridDim.x * 256 * U) {
        unsigned long long key[U][W], z[U], e[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int w = 0; w < W; ++w) key[u][w] = i0 + 32 * u < n ? keys[(i0 + 32 * u) * W + w] : 0ull;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            z[u] = aligned_z<W>(key[u], k);
            e[u] = i0 + 32 * u < n ? table[z[u] >> sh] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned long long p = i0 + 32 * u;
            unsigned long long s = z[u] >> sh;
            const unsigned fp = (unsigned)(mix_z(z[u]) >> 32);
            for (unsigned long long probe = 0; e[u] != 0ull && probe < cap; ++probe) {
                if ((unsigned)(e[u] >> 32) == fp) {
                    const unsigned long long i = (unsigned)e[u] - 1u;
                    bool same = true;
#pragma unroll
                    for (int w = 0; w < W; ++w) same = same && canon[i * W + w] == key[u][w];
                    if (same) {
                        kmer_record* r = out + i;  // `flipped` is already there
                        r->count = count[p];
#pragma unroll
                        for (int x = 0; x < 8; ++x) r->ext[x] = ext[p * 8 + x];
                        r->cls[0] = cls[2 * p];
                        r->cls[1] = cls[2 * p + 1];
                        r->found = 1;
                    }
                }
                s = (s + 1) & (cap - 1);
                e[u] = table[s];
            }
        }
    }
}

// The records of k-mers given before: the first one's, each with its own `flipped`.
__global__ void __launch_bounds__(256) wanted_repeat_kernel(const unsigned* __restrict__ rep, unsigned long long n,
                                                            kmer_record* out) {
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * 256) {
        const unsigned j = rep[i];
        if (j == (unsigned)i) continue;
        kmer_record r = out[j];
        r.flipped = out[i].flipped;
        out[i] = r;
    }
}

// Merge of Algorithm 1 (Sec. II-G): every k-mer of a second set (the
// contigs' k-mers, canonical and distinct) that is not among the survivors
// is appended to the survivors with count 0, zero tallies and its own
// classes; one that is already there keeps the survivor's record (the two
// occurrences collapse into one).  The index covers the survivors present
// before the merge; `n_out` counts appended positions (one reservation per
// warp).
template <int W>
__global__ void __launch_bounds__(256) merge_append_kernel(const unsigned long long* __restrict__ bkeys,
                                                           const unsigned char* __restrict__ bcls,
                                                           unsigned long long bn, unsigned k,
                                                           const unsigned* __restrict__ idx,
                                                           unsigned long long cap, unsigned long long* keys,
                                                           unsigned* count, unsigned* ext, unsigned char* cls,
                                                           unsigned long long out_cap,
                                                           unsigned long long* __restrict__ n_out,
                                                           unsigned* __restrict__ status) {
    const int lane = threadIdx.x & 31;
    const unsigned long long stride = (unsigned long long)gridDim.x * 256;
    for (unsigned long long base = blockIdx.x * 256ull + (threadIdx.x & ~31u); base < bn; base += stride) {
        const unsigned long long i = base + lane;
        bool add = false;
        unsigned long long key[W];
        if (i < bn) {
#pragma unroll
            for (int w = 0; w < W; ++w) key[w] = bkeys[i * W + w];
            add = true;
            unsigned long long s = index_home<W>(key, k, cap);
            for (unsigned long long probe = 0; probe < cap; ++probe) {
                const unsigned p = idx[s];
                if (p == kIdxEmpty) break;
                bool same = true;
#pragma unroll
                for (int w = 0; w < W; ++w) same = same && keys[(unsigned long long)p * W + w] == key[w];
                if (same) {
                    add = false;
                    break;
                }
                s = (s + 1) & (cap - 1);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, add);
        unsigned long long first = 0;
        if (lane == 0 && m) first = atomicAdd(n_out, (unsigned long long)__popc(m));
        first = __shfl_sync(0xffffffffu, first, 0);
        if (add) {
            const unsigned long long pos = first + __popc(m & ((1u << lane) - 1u));
            if (pos >= out_cap) {
                atomicOr(status, 1u);
            } else {
#pragma unroll
                for (int w = 0; w < W; ++w) keys[pos * W + w] = key[w];
                count[pos] = 0;
                uint4* eo = reinterpret_cast<uint4*>(ext + pos * 8);
                eo[0] = make_uint4(0, 0, 0, 0);
                eo[1] = make_uint4(0, 0, 0, 0);
                cls[2 * pos] = bcls[2 * i];
                cls[2 * pos + 1] = bcls[2 * i + 1];
            }
        }
    }
}

static unsigned grid_of(unsigned long long n, int num_sms) {
    unsigned long long g = (n + 255) / 256, cap = (unsigned long long)num_sms * 8;
    if (g > cap) g = cap;
    return g ? (unsigned)g : 1u;
}

cudaError_t launch_index_build(unsigned W, const unsigned long long* keys, unsigned long long n, unsigned k,
                               unsigned* idx, unsigned long long cap, int num_sms, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const unsigned g = grid_of(n, num_sms);
    switch (W) {
        case 1: index_build_kernel<1><<<g, 256, 0, s>>>(keys, n, k, idx, cap); break;
        case 2: index_build_kernel<2><<<g, 256, 0, s>>>(keys, n, k, idx, cap); break;
        case 3: index_build_kernel<3><<<g, 256, 0, s>>>(keys, n, k, idx, cap); break;
        case 4: index_build_kernel<4><<<g, 256, 0, s>>>(keys, n, k, idx, cap); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Cutting of contigs into pieces of `piece` bases that overlap by `lap`: a
// contig of L bases gives 1 + ceil((L - piece) / (piece - lap)) pieces (one if
// L <= piece), every one but the last of `piece` bases.
// count[c], bytes[c]: pieces of contig c and their bases; *bad counts
// contigs whose offsets decrease.
__global__ void __launch_bounds__(256) piece_count_kernel(const unsigned long long* __restrict__ off,
                                                          unsigned long long n, unsigned long long piece,
                                                          unsigned long long lap, unsigned long long* __restrict__ count,
                                                          unsigned long long* __restrict__ bytes,
                                                          unsigned long long* __restrict__ bad) {
    for (unsigned long long c = blockIdx.x * 256ull + threadIdx.x; c < n; c += (unsigned long long)gridDim.x * 256) {
        const unsigned long long a = off[c], e = off[c + 1];
        if (e < a) {
            atomicAdd(bad, 1ull);
            count[c] = bytes[c] = 0;
            continue;
        }
        const unsigned long long L = e - a, extra = L > piece ? (L - piece + (piece - lap) - 1) / (piece - lap) : 0ull;
        count[c] = extra + 1;
        bytes[c] = L + extra * lap;
    }
}

// Source and destination of every piece, from the scanned counts (pstart) and
// bases (bstart): n_pieces threads, each finding its contig by binary search.
__global__ void __launch_bounds__(256) piece_fill_kernel(const unsigned long long* __restrict__ off,
                                                         unsigned long long n, unsigned long long piece,
                                                         unsigned long long lap,
                                                         const unsigned long long* __restrict__ pstart,
                                                         const unsigned long long* __restrict__ bstart,
                                                         unsigned long long n_pieces,
                                                         unsigned long long* __restrict__ psrc,
                                                         unsigned long long* __restrict__ pdst) {
    for (unsigned long long p = blockIdx.x * 256ull + threadIdx.x; p < n_pieces; p += (unsigned long long)gridDim.x * 256) {
        unsigned long long lo = 0, hi = n;  // pstart[lo] <= p < pstart[hi]
        while (hi - lo > 1) {
            const unsigned long long mid = (lo + hi) / 2;
            if (pstart[mid] <= p) lo = mid; else hi = mid;
        }
        const unsigned long long i = p - pstart[lo];
        psrc[p] = off[lo] + i * (piece - lap);
        pdst[p] = bstart[lo] + i * piece;
        if (p == n_pieces - 1) pdst[n_pieces] = bstart[n];
    }
}

cudaError_t launch_piece_count(const unsigned long long* off, unsigned long long n, unsigned long long piece,
                               unsigned long long lap, unsigned long long* count, unsigned long long* bytes,
                               unsigned long long* bad, int num_sms, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    piece_count_kernel<<<grid_of(n, num_sms), 256, 0, s>>>(off, n, piece, lap, count, bytes, bad);
    return cudaGetLastError();
}

cudaError_t launch_piece_fill(const unsigned long long* off, unsigned long long n, unsigned long long piece,
                              unsigned long long lap, const unsigned long long* pstart,
                              const unsigned long long* bstart, unsigned long long n_pieces, unsigned long long* psrc,
                              unsigned long long* pdst, int num_sms, cudaStream_t s) {
    if (n_pieces == 0) return cudaSuccess;
    piece_fill_kernel<<<grid_of(n_pieces, num_sms), 256, 0, s>>>(off, n, piece, lap, pstart, bstart, n_pieces, psrc, pdst);
    return cudaGetLastError();
}

// Bytes of piece i: src[psrc[i] .. psrc[i] + (pdst[i + 1] - pdst[i])) copied
// to dst[pdst[i] ..); one CTA per piece at a time.
__global__ void __launch_bounds__(256) piece_copy_kernel(const char* __restrict__ src,
                                                         const unsigned long long* __restrict__ psrc,
                                                         const unsigned long long* __restrict__ pdst,
                                                         unsigned long long n_pieces, char* __restrict__ dst) {
    for (unsigned long long i = blockIdx.x; i < n_pieces; i += gridDim.x) {
        const unsigned long long a = psrc[i], b0 = pdst[i], len = pdst[i + 1] - b0;
        for (unsigned long long j = threadIdx.x; j < len; j += 256) dst[b0 + j] = src[a + j];
    }
}

cudaError_t launch_piece_copy(const char* src, const unsigned long long* psrc, const unsigned long long* pdst,
                              unsigned long long n_pieces, char* dst, int num_sms, cudaStream_t s) {
    if (n_pieces == 0) return cudaSuccess;
    const unsigned long long g = n_pieces < (unsigned long long)num_sms * 16 ? n_pieces : (unsigned long long)num_sms * 16;
    piece_copy_kernel<<<(unsigned)g, 256, 0, s>>>(src, psrc, pdst, n_pieces, dst);
    return cudaGetLastError();
}

cudaError_t launch_merge_append(unsigned W, const unsigned long long* bkeys, const unsigned char* bcls,
                                unsigned long long bn, unsigned k, const unsigned* idx, unsigned long long cap,
                                unsigned long long* keys, unsigned* count, unsigned* ext, unsigned char* cls,
                                unsigned long long out_cap, unsigned long long* n_out, unsigned* status, int num_sms,
                                cudaStream_t s) {
    if (bn == 0) return cudaSuccess;
    const unsigned g = grid_of(bn, num_sms);
    switch (W) {
        case 1: merge_append_kernel<1><<<g, 256, 0, s>>>(bkeys, bcls, bn, k, idx, cap, keys, count, ext, cls, out_cap, n_out, status); break;
        case 2: merge_append_kernel<2><<<g, 256, 0, s>>>(bkeys, bcls, bn, k, idx, cap, keys, count, ext, cls, out_cap, n_out, status); break;
        case 3: merge_append_kernel<3><<<g, 256, 0, s>>>(bkeys, bcls, bn, k, idx, cap, keys, count, ext, cls, out_cap, n_out, status); break;
        case 4: merge_append_kernel<4><<<g, 256, 0, s>>>(bkeys, bcls, bn, k, idx, cap, keys, count, ext, cls, out_cap, n_out, status); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

static unsigned long long wanted_slots(unsigned long long n) {
    unsigned long long cap = 1024;
    while (cap < 2 * n) cap <<= 1;
    return cap;
}

// The table, the canonical k-mers and who answers for each.
size_t wanted_scratch_bytes(unsigned W, unsigned long long n) { return wanted_slots(n) * 8 + n * 8 * W + n * 4; }

template <int W>
static cudaError_t launch_wanted_w(const unsigned long long* q, unsigned long long n, unsigned k, void* scratch,
                                   const unsigned long long* keys, const unsigned* count, const unsigned* ext,
                                   const unsigned char* cls, unsigned long long n_out, kmer_record* out, int num_sms,
                                   cudaStream_t s) {
    const unsigned long long cap = wanted_slots(n);
    unsigned long long* table = static_cast<unsigned long long*>(scratch);
    unsigned long long* canon = table + cap;
    unsigned* rep = reinterpret_cast<unsigned*>(canon + n * W);
    cudaError_t e = cudaMemsetAsync(table, 0, cap * 8, s);
    if (e != cudaSuccess) return e;
    wanted_build_kernel<W><<<grid_of(n, num_sms), 256, 0, s>>>(q, n, k, canon, table, cap, rep, out);
    if (n_out)
        wanted_stream_kernel<W><<<grid_of((n_out + 3) / 4, num_sms), 256, 0, s>>>(keys, n_out, k, canon, table, cap,
                                                                                  count, ext, cls, out);
    wanted_repeat_kernel<<<grid_of(n, num_sms), 256, 0, s>>>(rep, n, out);
    return cudaGetLastError();
}

cudaError_t launch_wanted(unsigned W, const unsigned long long* q, unsigned long long n, unsigned k, void* scratch,
                          const unsigned long long* keys, const unsigned* count, const unsigned* ext,
                          const unsigned char* cls, unsigned long long n_out, kmer_record* out, int num_sms,
                          cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    switch (W) {
        case 1: return launch_wanted_w<1>(q, n, k, scratch, keys, count, ext, cls, n_out, out, num_sms, s);
        case 2: return launch_wanted_w<2>(q, n, k, scratch, keys, count, ext, cls, n_out, out, num_sms, s);
        case 3: return launch_wanted_w<3>(q, n, k, scratch, keys, count, ext, cls, n_out, out, num_sms, s);
        case 4: return launch_wanted_w<4>(q, n, k, scratch, keys, count, ext, cls, n_out, out, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_lookup(unsigned W, const unsigned long long* q, unsigned long long n, unsigned k,
                          const unsigned* idx, unsigned long long cap, const unsigned long long* keys,
                          const unsigned* count, const unsigned* ext, const unsigned char* cls, kmer_record* out,
                          int num_sms, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const unsigned g = grid_of(n, num_sms);
    switch (W) {
        case 1: lookup_kernel<1><<<g, 256, 0, s>>>(q, n, k, idx, cap, keys, count, ext, cls, out); break;
        case 2: lookup_kernel<2><<<g, 256, 0, s>>>(q, n, k, idx, cap, keys, count, ext, cls, out); break;
        case 3: lookup_kernel<3><<<g, 256, 0, s>>>(q, n, k, idx, cap, keys, count, ext, cls, out); break;
        case 4: lookup_kernel<4><<<g, 256, 0, s>>>(q, n, k, idx, cap, keys, count, ext, cls, out); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace kmer
