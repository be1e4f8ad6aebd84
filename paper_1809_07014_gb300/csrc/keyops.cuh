// Operations on canonical k-mer keys held as W 64-bit words (word 0 most
// significant, holding the first 2k - 64(W-1) bits): base access, the
// survivors' index (an open-addressing table of survivor positions), and the
// shifts that step from a k-mer to its neighbours in the de Bruijn graph.
#pragma once
#include "common.cuh"

namespace kmer {

constexpr unsigned kIdxEmpty = 0xFFFFFFFFu;

// z of a key (common.cuh), left-aligned: its top bits are the key's partition.
template <int W>
__device__ __forceinline__ unsigned long long aligned_z(const unsigned long long (&key)[W], unsigned k) {
    const unsigned bt = W == 1 ? 2 * k : 64;
    return key_to_z<W>(key, bt) << (64 - bt);
}
__device__ __forceinline__ unsigned long long mix_z(unsigned long long z) {
    z ^= z >> 29;
    return z * 0xFF51AFD7ED558CCDull;
}

// Home slot of a key in the survivors' index of `cap` slots (a power of two, at
// least 1024): which 64th of the index from the top bits of z, the place in
// it from a mix of z.  Survivors come out partition by partition, so that a
// build, or lookups of another analysis's k-mers, stay in one 64th at a time
// (16 MB of 1 GB, in L2), while the slots of one moment lie apart (with the
// top bits alone the neighbours' claims meet in the same lines: 101 M one-word
// survivors indexed in 3.7-5.2 ms, against 4.0 this way and 4.3 with an
// unrelated hash; the merge's lookups of 15 M k-mers: 0.70-0.88 ms unrelated,
// 0.48 this way).
template <int W>
__device__ __forceinline__ unsigned long long index_home(const unsigned long long (&key)[W], unsigned k,
                                                         unsigned long long cap) {
    constexpr unsigned kHi = 6;
    const unsigned long long z = aligned_z<W>(key, k);
    const unsigned lc = 63u - __clzll((long long)cap);
    return ((z >> (64 - kHi)) << (lc - kHi)) | ((mix_z(z) >> 32) & ((cap - 1) >> kHi));
}

// Base i (0 = first, most significant) of a k-mer held as W words, word 0
// most significant.
template <int W>
__device__ __forceinline__ unsigned get_base(const unsigned long long (&key)[W], unsigned k, unsigned i) {
    const unsigned pos = 2 * (k - 1 - i);  // bit position from the least significant end
    return (unsigned)(key[W - 1 - pos / 64] >> (pos % 64)) & 3u;
}

// Position of `key` among the survivors through the index, or kIdxEmpty.
template <int W>
__device__ __forceinline__ unsigned index_find(const unsigned long long (&key)[W], unsigned k,
                                               const unsigned* __restrict__ idx, unsigned long long cap, const unsigned long long* __restrict__ keys) {
    unsigned long long s = index_home<W>(key, k, cap);
    for (unsigned long long probe = 0; probe < cap; ++probe) {
        const unsigned p = idx[s];
        if (p == kIdxEmpty) return kIdxEmpty;
        bool same = true;
#pragma unroll
        for (int w = 0; w < W; ++w) same = same && keys[(unsigned long long)p * W + w] == key[w];
        if (same) return p;
        s = (s + 1) & (cap - 1);
    }
    return kIdxEmpty;
}

// The k-mer shifted one base to the left with base b appended (the right
// neighbour's string); hb = bits of word 0.
template <int W>
__device__ __forceinline__ void shift_in_right(unsigned long long (&x)[W], unsigned b, unsigned hb) {
#pragma unroll
    for (int w = 0; w < W - 1; ++w) x[w] = (x[w] << 2) | (x[w + 1] >> 62);
    x[W - 1] = (x[W - 1] << 2) | b;
    x[0] &= low_mask(hb);
}

// The k-mer shifted one base to the right with base b put first (the left
// neighbour's string).
template <int W>
__device__ __forceinline__ void shift_in_left(unsigned long long (&x)[W], unsigned b, unsigned hb) {
#pragma unroll
    for (int w = W - 1; w > 0; --w) x[w] = (x[w] >> 2) | (x[w - 1] << 62);
    x[0] = (x[0] >> 2) | ((unsigned long long)b << (hb - 2));
}

// Whole words: the bases of each reversed and complemented by bit reversal,
// then all moved down by the unused bits of word 0 (which uses hb, 2 to 62 for
// odd k).
template <int W>
__device__ __forceinline__ void reverse_complement(const unsigned long long (&x)[W], unsigned k,
                                                   unsigned long long (&rc)[W]) {
    const unsigned hb = 2 * k - 64 * (W - 1);
    unsigned long long r[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const unsigned long long m = __brevll(~x[W - 1 - w]);
        r[w] = ((m >> 1) & 0x5555555555555555ull) | ((m & 0x5555555555555555ull) << 1);
    }
    rc[0] = r[0] >> (64 - hb);
#pragma unroll
    for (int w = 1; w < W; ++w) rc[w] = (r[w - 1] << hb) | (r[w] >> (64 - hb));
}

// a < b, word 0 first (lexicographic order of the k-mers).
template <int W>
__device__ __forceinline__ bool key_less(const unsigned long long (&a)[W], const unsigned long long (&b)[W]) {
#pragma unroll
    for (int w = 0; w < W; ++w)
        if (a[w] != b[w]) return a[w] < b[w];
    return false;
}

}  // namespace kmer
