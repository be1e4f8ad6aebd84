// Steps a2 + a3: slide a k-window over one packed read, keep the forward
// k-mer and its reverse complement as W-word shift registers, and produce for
// every window without N its canonical key (the smaller of the two) and its
// extension code.  Sec. II-B: k-mers overlap by k-1 bases; the extensions are
// the bases just before and after the window in the read, kept only if they
// are A/C/G/T with Phred >= threshold (the pack step folded both tests into
// one "good" bit per base).
#pragma once
#include "common.cuh"

namespace kmer {

// A window's words a < b, word 0 most significant: one borrow chain, no branch.
template <int W>
__device__ __forceinline__ bool words_less(const unsigned long long (&a)[W], const unsigned long long (&b)[W]) {
    if constexpr (W == 1) {
        return a[0] < b[0];
    } else {
        unsigned r;
        unsigned long long t;
        if constexpr (W == 2)
            asm("sub.cc.u64 %1, %2, %4;\n\tsubc.cc.u64 %1, %3, %5;\n\tsubc.u32 %0, 0, 0;"
                : "=r"(r), "=&l"(t) : "l"(a[1]), "l"(a[0]), "l"(b[1]), "l"(b[0]));
        else if constexpr (W == 3)
            asm("sub.cc.u64 %1, %2, %5;\n\tsubc.cc.u64 %1, %3, %6;\n\tsubc.cc.u64 %1, %4, %7;\n\tsubc.u32 %0, 0, 0;"
                : "=r"(r), "=&l"(t) : "l"(a[2]), "l"(a[1]), "l"(a[0]), "l"(b[2]), "l"(b[1]), "l"(b[0]));
        else
            asm("sub.cc.u64 %1, %2, %6;\n\tsubc.cc.u64 %1, %3, %7;\n\tsubc.cc.u64 %1, %4, %8;\n\t"
                "subc.cc.u64 %1, %5, %9;\n\tsubc.u32 %0, 0, 0;"
                : "=r"(r), "=&l"(t)
                : "l"(a[3]), "l"(a[2]), "l"(a[1]), "l"(a[0]), "l"(b[3]), "l"(b[2]), "l"(b[1]), "l"(b[0]));
        return r != 0u;
    }
}

// The 32 bases of a word reversed and complemented.
__device__ __forceinline__ unsigned long long revcomp_word(unsigned long long x) {
    const unsigned long long m = __brevll(~x);
    return ((m >> 1) & 0x5555555555555555ull) | ((m & 0x5555555555555555ull) << 1);
}

// One read's windows in order, from any window on.  init() stands at window
// w0: its words come from the packed blocks by shifts, its reverse complement
// by bit reversal and the last N before it from the N masks, so the k bases
// of the first window cost no steps (two thirds of a 150-base read's steps at
// k = 99, a fifth at k = 31), and several threads can share a read.
//
// HI (one word, k >= 17): the window's first base sits in the high 32 bits
// of the word, so the base leaving the window and the complement entering the
// reverse strand touch that half only.
template <int W, bool HI = false>
struct Roll {
    unsigned long long fwd[W], rc[W];
    unsigned long long cur;        // bases of the current block, next base in the top 2 bits
    unsigned curn, curg;           // N / good bits of the current block, next base in bit 0
    unsigned lg, lgn;              // good bits of the bases that left the window, next in bit 0; the block after
    uint4 nxt;                     // the block after the current one, loaded one block ahead
    unsigned out;                  // base that left the window at the last step
    unsigned L, k, sh;             // sh: shift of the window's first base within its 32-bit half
    unsigned first_ok;             // first step whose window holds no N: last N position + k + 1
    const PackedBlock* blk;
    unsigned long long mask;       // bits of word 0

    // Stands before step k + w0, at the window of bases [w0, w0 + k); a read
    // without that window (w0 + k > L) has no steps.
    __device__ void init(const Job& j, unsigned long long r, unsigned w0 = 0) {
        const unsigned long long a = j.offsets[r];
        L = (unsigned)(j.offsets[r + 1] - a);  // reads are shorter than 2^31 bases
        blk = j.blocks + j.blk_off[r];
        k = j.g.k;
        const unsigned hb = j.g.hb;
        mask = low_mask(hb);
        sh = hb - 2;
        const unsigned t = w0 + k;
        first_ok = t;
        out = lg = lgn = 0;
        cur = 0;
        curn = curg = 0;
        nxt = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int i = 0; i < W; ++i) fwd[i] = rc[i] = 0;
        if (t > L) return;
        // A[i]: the 32 bases from w0 + 32 i on, from two blocks (none past the read's last)
        const unsigned b0 = w0 >> 5, o = w0 & 31u, o2 = 2 * o;
        const unsigned blocks = (L + 31) / 32;
        const uint4 none = make_uint4(0, 0, 0, 0);
        uint4 x = __ldg(reinterpret_cast<const uint4*>(blk + b0));
        if (o == 0) lgn = x.w;
        else lg = x.w >> (o - 1);  // base w0 - 1 next
        if (w0) {
            const uint4 y = o ? x : __ldg(reinterpret_cast<const uint4*>(blk + b0 - 1));
            if (!o) lg = y.w >> 31;
            const unsigned at = (w0 - 1) & 31u;
            out = (unsigned)((((unsigned long long)y.y << 32 | y.x) >> (62 - 2 * at)) & 3ull);
        }
        unsigned long long A[W];
        unsigned last_n = 0;  // last N of the window, plus one, from w0
        const unsigned rest = k - 32 * (W - 1);  // 1..31 bases of the last word (k odd)
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const bool more = b0 + i + 1 < blocks;
            const uint4 y = more ? __ldg(reinterpret_cast<const uint4*>(blk + b0 + i + 1)) : none;
            if (i == 0 && o) lgn = y.w;
            const unsigned long long bx = (unsigned long long)x.y << 32 | x.x, by = (unsigned long long)y.y << 32 | y.x;
            A[i] = o ? (bx << o2) | (by >> (64 - o2)) : bx;
            unsigned nm = __funnelshift_r(x.z, y.z, o);
            if (i == W - 1) nm &= (1u << rest) - 1u;
            if (nm) last_n = 32 * i + 32 - __clz(nm);
            if (i == W - 1) {  // base t is in this block or the next
                const unsigned ot = t & 31u;
                const bool same = t >> 5 == b0 + i;
                const uint4 c = same ? x : y;
                cur = ((unsigned long long)c.y << 32 | c.x) << (2 * ot);
                curn = c.z >> ot;
                curg = c.w >> ot;
                // the block after base t's; step t takes nxt when t starts a block
                const unsigned nb = ot ? (t >> 5) + 1 : t >> 5;
                nxt = nb < blocks ? __ldg(reinterpret_cast<const uint4*>(blk + nb)) : none;
            }
            x = y;
        }
        if (last_n) first_ok = w0 + last_n + k;
        fwd[0] = A[0] >> (64 - hb);
#pragma unroll
        for (int i = 1; i < W; ++i) fwd[i] = (A[i - 1] << hb) | (A[i] >> (64 - hb));
        unsigned long long R[W];
#pragma unroll
        for (int i = 0; i < W; ++i) R[i] = revcomp_word(fwd[W - 1 - i]);
        rc[0] = R[0] >> (64 - hb);
#pragma unroll
        for (int i = 1; i < W; ++i) rc[i] = (R[i - 1] << hb) | (R[i] >> (64 - hb));
    }

    // Step t = w0 + k, w0 + k + 1, ..., L, in order.  First the window [t-k, t) is
    // reported if it holds no N; then base t (if t < L) is shifted in.
    // Returns true and fills key / lcode / rcode (0 = none, 1..4 = A..T) for a
    // window.
    __device__ __forceinline__ bool step(unsigned t, unsigned long long (&key)[W], unsigned& lcode, unsigned& rcode) {
        const bool in = t < L;
        unsigned b = 0, good = 0, isn = 0;
        if (in) {
            if ((t & 31) == 0) {
                cur = ((unsigned long long)nxt.y << 32) | nxt.x;
                curn = nxt.z;
                curg = nxt.w;
                if (t + 32 < L) nxt = __ldg(reinterpret_cast<const uint4*>(blk + (t >> 5) + 1));
            }
            b = (unsigned)(cur >> 62);
            cur <<= 2;
            isn = curn & 1u;
            curn >>= 1;
            good = curg & 1u;
            curg >>= 1;
        }
        // the base before the window, t - k - 1: none at the first step (lg starts at 0);
        // base q = t - k leaves the window now and is next in lg
        const unsigned lgood = lg & 1u;
        const unsigned q = t - k;
        if ((q & 31) == 0) {
            lg = lgn;
            if (q + 32 < L) lgn = __ldg(&blk[(q >> 5) + 1].hqmask);
        } else {
            lg >>= 1;
        }
        const bool emit = t >= first_ok;
        if (emit) {
            unsigned lc = lgood ? out + 1 : 0;
            unsigned rcd = good ? b + 1 : 0;
            // canonical: the lexicographically smaller of forward and reverse complement
            const bool flip = words_less<W>(rc, fwd);
#pragma unroll
            for (int w = 0; w < W; ++w) key[w] = flip ? rc[w] : fwd[w];
            if (flip) {  // the key reads the other strand: swap sides, complement bases
                const unsigned nl = rcd ? 5 - rcd : 0, nr = lc ? 5 - lc : 0;
                lc = nl;
                rcd = nr;
            }
            lcode = lc;
            rcode = rcd;
        }
        if (in) {
            if (HI) {
                out = ((unsigned)(fwd[0] >> 32) >> (sh - 32)) & 3u;
            } else {
                out = (unsigned)(fwd[0] >> sh) & 3u;
            }
#pragma unroll
            for (int w = 0; w < W - 1; ++w) fwd[w] = (fwd[w] << 2) | (fwd[w + 1] >> 62);
            fwd[W - 1] = (fwd[W - 1] << 2) | b;
            fwd[0] &= mask;
#pragma unroll
            for (int w = W - 1; w > 0; --w) rc[w] = (rc[w] >> 2) | (rc[w - 1] << 62);
            rc[0] = (rc[0] >> 2) | (HI ? (unsigned long long)((3u - b) << (sh - 32)) << 32 : (unsigned long long)(3u - b) << sh);
            if (isn) first_ok = t + k + 1;
        }
        return emit;
    }
};

// Record of one window (words 0..W-2 = head words, word W-1 = tail) and its
// level-1 bucket; returns false when the window belongs to another pass.
template <int W>
__device__ __forceinline__ bool make_record(const Geometry& g, unsigned pass, const unsigned long long (&key)[W],
                                            unsigned lcode, unsigned rcode, unsigned long long (&rec)[W],
                                            unsigned& bucket) {
    const unsigned long long z = key_to_z<W>(key, g.bt);
    if (g.ps && (unsigned)(z >> (g.bt - g.ps)) != pass) return false;
    const unsigned zb = g.zl_bits();
    bucket = g.p1 ? (unsigned)(z >> zb) & ((1u << g.p1) - 1u) : 0u;
#pragma unroll
    for (int w = 0; w < W - 1; ++w) rec[w] = key[w];
    rec[W - 1] = ((z & low_mask(zb)) << 6) | ext_code(lcode, rcode);
    return true;
}

// Bloom-gate hash of a canonical key (gate.cu): the 64-bit finaliser of
// MurmurHash3 applied to the last word xored with a hash of the head words.
template <int W>
__device__ __forceinline__ unsigned long long gate_hash(const unsigned long long (&key)[W]) {
    unsigned long long h = key[W - 1] ^ head_hash<W>(key) ^ 0x2545F4914F6CDD1Dull;
    h ^= h >> 33;
    h *= 0xFF51AFD7ED558CCDull;
    h ^= h >> 33;
    h *= 0xC4CEB9FE1A85EC53ull;
    h ^= h >> 33;
    return h;
}

// The filter word (the hash's share of `words`, from its top bits) and four
// bits within it (four 6-bit fields of the low bits).
struct GateProbe {
    unsigned long long word, mask;
};
__device__ __forceinline__ GateProbe gate_probe(unsigned long long h, unsigned long long words) {
    GateProbe p;
    p.word = __umul64hi(h, words);
    p.mask = (1ull << (h & 63)) | (1ull << ((h >> 6) & 63)) | (1ull << ((h >> 12) & 63)) | (1ull << ((h >> 18) & 63));
    return p;
}

// The key is in the gate's filter (every bit of its probe set).
template <int W>
__device__ __forceinline__ bool gate_has(const unsigned long long* f, unsigned long long words,
                                         const unsigned long long (&key)[W]) {
    const GateProbe p = gate_probe(gate_hash<W>(key), words);
    return (__ldg(f + p.word) & p.mask) == p.mask;
}

// z of a record held in a known pass and level-1 bucket.
__device__ __forceinline__ unsigned long long record_z(const Geometry& g, unsigned pass, unsigned bucket,
                                                       unsigned long long tail) {
    const unsigned zb = g.zl_bits();
    unsigned long long z = tail >> 6;
    if (g.p1) z |= (unsigned long long)bucket << zb;
    if (g.ps) z |= (unsigned long long)pass << (g.bt - g.ps);
    return z;
}

}  // namespace kmer
