// Steps a4-a7 fused: each leaf (partition) is counted in a shared-memory
// open-addressing table (the owner-local histogram of Sec. II-A use case 4,
// with the per-k-mer count and left/right extension tallies of Sec. II-B),
// then the table is swept once: k-mers below min_count are dropped, both
// sides are classified (Sec. II-C) and survivors are compacted to the output
// arrays.
//
// Persistent CTAs walk the leaves; while one leaf is being swept, the first
// batch of the next leaf's records is already loading into registers.
//
// Table (shared memory, planes of `cap_max` entries, a leaf uses the first
// `cap` slots): the tail word of each slot (0 = empty; else the tail of the
// record that claimed the slot, plus one: its key and that record's extension
// code), W-1 head words (two-word keys keep tail and head side by side, one
// 16-byte pair per slot claimed by a 128-bit CAS), and nine 16-bit tallies of
// the other records, packed in five 32-bit planes: left A, C, G, T, "no left
// extension" (so that count = one + the five left lanes and needs no counter
// of its own), right A, C, G, T.  Slots are probed in groups of 16 bytes of
// keys (two tails, or one two-word key), a key's groups a hashed step apart.
// A leaf with 65536 records or more (where a 16-bit tally could wrap) is
// recounted exactly by the HBM-table fallback; one whose keys do not fit its
// table is counted again in key ranges (leaf_split_kernel).
//
// What bounds it: latency of the probe rounds and the issue slots (about 0.67
// instructions a cycle and scheduler, half of the shared-memory pipe), not
// DRAM.  On the 2-Gbase reads at k = 31 (1.6 G records, 508 M keys) 18.5 ->
// 13.6 ms, at k = 99 (103 M records, 89 M keys) 5.3 -> 3.7 ms, from: the
// claiming record keeping its extension code in the slot (no tally for a third
// of the records at k = 31, for six in seven at k = 99; most k-mers are seen
// once), hashed steps between groups (consecutive groups clustered: leaves
// above 0.6 of a table overflowed their probe limit), 32-bit shared-memory
// addresses, one-word probe rounds of full warps (a queue per warp: 14.4 ->
// 13.6 ms), job fields in shared memory instead of global loads in the sweep,
// four slots per lane in the sweep, and fuller leaves (0.75 of a table).
//
// Every plane is zero between leaves: the sweep clears each slot after
// reading it, so no separate clearing pass is needed.
#include "kernels.h"
#include "roll.cuh"

namespace kmer {

constexpr int kLeafThreads = 512;
constexpr int kLeafWarps = kLeafThreads / 32;
constexpr unsigned kLeafFull = 1u, kLeafTimeout = 4u;
constexpr unsigned kSpinLimit = 1u << 22;
constexpr unsigned kMaxRounds = 64;       // probe rounds of one record; past them the leaf goes to its key ranges
constexpr unsigned kLanePlanes = 5;
constexpr unsigned kMaxSubBits = 4;       // a leaf is split into at most 16 key ranges
// Slot tail of an occupied key: the tail of the record that claimed it plus
// one, so that its low six bits hold that record's extension code + 1 (at most
// 37, never 0; 0 = empty slot).  The claiming record needs no tally of its own.
// kBusy in those bits marks a slot being published (W > 2).
constexpr unsigned kBusy = 63u;

template <int W>
struct LeafShape {
    static constexpr int U = W == 1 ? 4 : 2;  // records per thread per batch
    static constexpr int B = U * kLeafThreads;
};

// One-word records that a probe round leaves unsettled wait in their warp's
// queue (the record and its probe state): up to 31 from before plus 32.
constexpr unsigned kQueue = 64;
__host__ __device__ inline size_t leaf_queue_bytes(unsigned W) { return W == 1 ? (size_t)kLeafWarps * kQueue * 12 : 0; }

// bytes per slot: tail, heads, 5 tally planes, survivor list entry
__host__ __device__ inline size_t leaf_slot_bytes(unsigned W) { return (size_t)8 * W + 4 * kLanePlanes + 2; }

size_t leaf_smem_bytes(unsigned W, unsigned cap) { return leaf_slot_bytes(W) * cap + leaf_queue_bytes(W) + 64; }

unsigned leaf_table_cap(unsigned W, size_t smem_budget) {
    size_t c = (smem_budget - 64 - leaf_queue_bytes(W)) / leaf_slot_bytes(W);
    return (unsigned)(c & ~63ull);  // a slice of a multiple of four slots per warp
}

struct LeafInfo {
    unsigned bucket;
    unsigned long long start, n;
    const unsigned long long* recs;
    bool ok;
};

__device__ __forceinline__ LeafInfo leaf_info(const Job& j, unsigned leaf) {
    LeafInfo li;
    unsigned long long capr;
    if (j.g.p2 == 0) {
        li.bucket = leaf;
        li.start = j.l1_start[leaf];
        li.n = j.l1_fill[leaf];
        capr = j.l1_cap[leaf];
        li.recs = j.l1_rec;
    } else {
        li.bucket = leaf >> j.g.p2;
        const unsigned sub = leaf & ((1u << j.g.p2) - 1u);
        if (j.l2_leaf_start) {
            li.start = j.l2_leaf_start[leaf];
            capr = j.l2_leaf_start[leaf + 1] - li.start;
        } else {
            li.start = j.l2_base[li.bucket] + (unsigned long long)sub * j.l2_leafcap[li.bucket];
            capr = j.l2_leafcap[li.bucket];
        }
        li.n = j.l2_fill[leaf];
        li.recs = j.l2_rec;
    }
    // an overfull leaf was reported by its writer and the host retries; skip it
    li.ok = li.n > 0 && li.n <= capr;
    return li;
}

template <int W>
__device__ __forceinline__ void load_batch(const LeafInfo& li, unsigned first,
                                           unsigned long long (&r)[LeafShape<W>::U][W]) {
    constexpr int U = LeafShape<W>::U;
    const unsigned long long* src = li.recs + li.start * W;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const unsigned i = first + u * kLeafThreads + threadIdx.x;
#pragma unroll
        for (int w = 0; w < W; ++w) r[u][w] = (li.ok && i < li.n) ? __ldcs(src + (size_t)i * W + w) : 0ull;
    }
}

// The table's planes as 32-bit shared-memory addresses (bytes): every access
// below is an explicit shared-memory instruction with a 32-bit address, so no
// address is computed in 64 bits.
struct Table {
    unsigned tail;    // 8 bytes a slot (two-word keys: 16, tail and head)
    unsigned heads;   // W - 1 planes of 8 bytes a slot
    unsigned lanes;   // 5 planes of 4 bytes a slot
    unsigned list;    // 2 bytes a slot
    unsigned queue;   // this warp's queue (one-word keys): kQueue records, then kQueue states
    unsigned stride;  // slots of a plane
};

__device__ __forceinline__ unsigned lds32(unsigned a) {
    unsigned v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long lds64(unsigned a) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128(unsigned a) {
    uint4 r;
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a) : "memory");
    return r;
}
// The keys of a probe group, which other warps may be claiming: two whole
// 64-bit words (a vector of 32-bit words would promise nothing about the halves
// of a tail), split in registers.
__device__ __forceinline__ uint4 lds_keys(unsigned a) {
    unsigned long long lo, hi;
    asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "r"(a) : "memory");
    return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}
__device__ __forceinline__ void sts32(unsigned a, unsigned v) {
    asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned lds16(unsigned a) {
    unsigned short v;
    asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts16(unsigned a, unsigned v) {
    asm volatile("st.volatile.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void sts64(unsigned a, unsigned long long v) {
    asm volatile("st.volatile.shared.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void sts128_zero(unsigned a) {
    asm volatile("st.volatile.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(0u) : "memory");
}
__device__ __forceinline__ void add_shared(unsigned a, unsigned v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// v replaces 0; returns the previous contents.
__device__ __forceinline__ unsigned long long claim64(unsigned a, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.shared.cas.b64 %0, [%1], %2, %3;" : "=l"(old) : "r"(a), "l"(0ull), "l"(v) : "memory");
    return old;
}
// {lo, hi} replaces {0, 0}; returns the previous contents.
__device__ __forceinline__ void claim128(unsigned a, unsigned long long lo, unsigned long long hi,
                                         unsigned long long& old_lo, unsigned long long& old_hi) {
    asm volatile(
        "{\n\t.reg .b128 cmp, val, old;\n\t"
        "mov.b128 cmp, {%4, %4};\n\t"
        "mov.b128 val, {%2, %3};\n\t"
        "atom.shared.cas.b128 old, [%5], cmp, val;\n\t"
        "mov.b128 {%0, %1}, old;\n\t}"
        : "=l"(old_lo), "=l"(old_hi)
        : "l"(lo), "l"(hi), "l"(0ull), "r"(a)
        : "memory");
}

// Tally lane q in 0..8 of a slot lives in plane q >> 1, half q & 1.
__device__ __forceinline__ void bump(const Table& t, unsigned slot, unsigned q) {
    add_shared(t.lanes + 4 * ((q >> 1) * t.stride + slot), q & 1u ? 0x10000u : 1u);
}

// Key words of a slot.  One-word keys: the tail plane.  Two-word keys:
// (tail, head) pairs, 16 bytes per slot over the first two planes, claimed
// whole by one 128-bit CAS.  Wider keys: the tail plane and W-1 head planes,
// published with a busy mark.
template <int W>
__device__ __forceinline__ unsigned long long slot_tail(const Table& t, unsigned s) {
    return lds64(t.tail + (W == 2 ? 16 : 8) * s);
}
template <int W>
__device__ __forceinline__ unsigned head_addr(const Table& t, unsigned w, unsigned s) {
    return W == 2 ? t.tail + 16 * s + 8 : t.heads + 8 * (w * t.stride + s);
}
// Probe groups of a table of `cap` slots: 16 bytes of keys each (two tails, or
// one two-word key), read by one shared-memory load.
template <int W>
__device__ __forceinline__ unsigned groups_of(unsigned cap) { return W == 2 ? cap : cap / 2; }

// A tail (lo, hi words) of an occupied slot is the key of tail k (the low six
// bits are the claiming record's extension code).
__device__ __forceinline__ bool same_tail(unsigned lo, unsigned hi, unsigned klo, unsigned khi) {
    return (((lo ^ klo) & ~63u) | (hi ^ khi)) == 0u && lo != 0u;
}

// A key goes through groups home, home + step, ... of the table.  The slots of
// a group fill in order and none empties while a leaf is counted, so a group's
// first empty slot is the number of occupied ones, and a claim there can only
// succeed when every slot before it holds a key that was compared: a key never
// gets two slots.  The record that claims a slot leaves its extension code
// there; the others add to the slot's tallies.
//
// Home group from every in-leaf bit of z (the low bits of z depend on few
// bits of the key, its top bits are the leaf's): a multiplicative hash.
__device__ __forceinline__ unsigned leaf_hash(unsigned long long tail) {
    return ((unsigned)tail & ~63u) * 0x9E3779B1u + (unsigned)(tail >> 32) * 0x85EBCA77u;
}
// Groups between one probe and the next: odd and below 256 (a table has 512
// groups or more).  The groups are a multiple of 32, so a key comes to 32
// different ones at least before it meets one again: to all 64 of its rounds
// unless the step shares a large odd factor with the number of groups.  Such a
// key may send its leaf to the key ranges early, which changes no result.
__device__ __forceinline__ unsigned leaf_step(unsigned hsh) { return (hsh >> 8 & 255u) | 1u; }

__device__ __forceinline__ void tally(const Table& t, unsigned slot, unsigned long long tail) {
    const unsigned l = ext_left(tail), r = ext_right(tail);
    bump(t, slot, l ? l - 1 : 4u);  // every counted window has exactly one left lane (the first: its code)
    if (r) bump(t, slot, 4u + r);
}

// One probe round of a warp (every lane calls; lanes with `have` hold a record
// that probes group g, `full` groups so far): one 16-byte load, at most one
// claim.  A record that is not settled (its group is full, or another key took
// the slot it tried) goes to the warp's queue, `waiting` records so far.
__device__ __forceinline__ void probe_round(const Table& t, const unsigned long long tail, bool have, unsigned g,
                                            unsigned full, unsigned hsh, unsigned ngroups, unsigned& waiting,
                                            unsigned* s_flags) {
    // the code's + 1 does not carry out of bit 5
    const unsigned klo = (unsigned)tail + 1u, khi = (unsigned)(tail >> 32);
    bool again = false;
    if (have) {
        const unsigned ga = t.tail + 16 * g;
        const uint4 a = lds_keys(ga);
        const bool e0 = same_tail(a.x, a.y, klo, khi), e1 = same_tail(a.z, a.w, klo, khi);
        bool hit = e0 || e1;
        unsigned slot = 2 * g + (e1 ? 1u : 0u);
        again = !hit;
        if (!hit && a.z == 0u) {
            const unsigned occ = a.x ? 1u : 0u;
            const unsigned long long old = claim64(ga + 8 * occ, tail + 1ull);
            slot = 2 * g + occ;
            hit = old != 0ull && same_tail((unsigned)old, (unsigned)(old >> 32), klo, khi);
            again = old != 0ull && !hit;  // another key took the slot: the group is read again
        } else if (!hit) {
            g += leaf_step(hsh);
            g -= g >= ngroups ? ngroups : 0u;
            ++full;
        }
        if (hit) tally(t, slot, tail);
        if (full >= kMaxRounds) {
            again = false;
            atomicOr(s_flags, kLeafFull);
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, again);
    if (again) {
        const unsigned at = waiting + __popc(m & ((1u << (threadIdx.x & 31u)) - 1u));
        sts64(t.queue + 8 * at, tail);
        sts32(t.queue + 8 * kQueue + 4 * at, full << 16 | g);  // g is below 65 536
    }
    waiting += __popc(m);
    __syncwarp();
}

// A probe round of the last (up to 32) records of the warp's queue.
__device__ __forceinline__ void probe_queue(const Table& t, unsigned ngroups, unsigned& waiting, unsigned* s_flags) {
    const unsigned n = waiting < 32u ? waiting : 32u, at = waiting - n + (threadIdx.x & 31u);
    const bool have = (threadIdx.x & 31u) < n;
    const unsigned long long tail = have ? lds64(t.queue + 8 * at) : 0ull;
    const unsigned state = have ? lds32(t.queue + 8 * kQueue + 4 * at) : 0u;
    __syncwarp();
    waiting -= n;
    probe_round(t, tail, have, state & 0xFFFFu, state >> 16, leaf_hash(tail), ngroups, waiting, s_flags);
}

// Two words and more: slot of a record's key, or kClaimed when the record
// claimed a new one, kNoSlot after kMaxRounds full groups, kGaveUp after a
// wait that gave up.  A lane leaves as soon as its record is settled: the
// lanes of a warp drift apart, which pays here (queued full-warp rounds as for
// one word, with either CAS, took 1.09 ms against 0.59 on 32 M two-word
// records) and not there (20.5 ms against 14.3 on 1.6 G).
constexpr int kClaimed = -1, kNoSlot = -2, kGaveUp = -3;

template <int W>
__device__ __forceinline__ int find_slot(const Table& t, const unsigned long long (&rec)[W], unsigned ngroups) {
    constexpr unsigned GS = W == 2 ? 1 : 2;  // slots of a group
    const unsigned lo = (unsigned)rec[W - 1], khi = (unsigned)(rec[W - 1] >> 32), klo = lo + 1u;
    const unsigned hsh = leaf_hash(rec[W - 1]);
    const unsigned long long ktail = rec[W - 1] + 1ull;
    unsigned g = __umulhi(hsh, ngroups);
    for (unsigned it = 0; it < kMaxRounds;) {
        const unsigned ga = t.tail + 16 * g;
        const uint4 a = lds_keys(ga);
        if constexpr (W == 2) {
            unsigned long long ct = (unsigned long long)a.y << 32 | a.x, ch = (unsigned long long)a.w << 32 | a.z;
            if (a.x == 0u) {  // empty, or still being claimed
                claim128(ga, ktail, rec[0], ct, ch);
                if (ct == 0ull && ch == 0ull) return kClaimed;
            }
            if (same_tail((unsigned)ct, (unsigned)(ct >> 32), klo, khi)) {
                // a plain read may catch a claim half done (the tail without its head):
                // another head is read again by a CAS that cannot change the slot
                if (ch != rec[0]) claim128(ga, 0ull, 0ull, ct, ch);
                if (ch == rec[0]) return (int)g;
            }
        } else {
            const unsigned occ = (a.x ? 1u : 0u) + (a.z ? 1u : 0u);
            for (unsigned s = 0; s < occ; ++s) {
                if (!same_tail(s ? a.z : a.x, s ? a.w : a.y, klo, khi)) continue;
                for (unsigned spins = 0; (lds32(ga + 8 * s) & 63u) == kBusy;)  // its heads are being written
                    if (++spins > kSpinLimit) return kGaveUp;
                __threadfence_block();
                bool same = true;
#pragma unroll
                for (int w = 0; w < W - 1; ++w) same = same && lds64(head_addr<W>(t, w, 2 * g + s)) == rec[w];
                if (same) return (int)(2 * g + s);
            }
            if (occ < GS) {
                if (claim64(ga + 8 * occ, ktail | kBusy) != 0ull) continue;  // taken: the group is read again
#pragma unroll
                for (int w = 0; w < W - 1; ++w) sts64(head_addr<W>(t, w, 2 * g + occ), rec[w]);
                __threadfence_block();
                sts64(ga + 8 * occ, ktail);
                return kClaimed;
            }
        }
        ++it;
        g += leaf_step(hsh);
        g -= g >= ngroups ? ngroups : 0u;
    }
    return kNoSlot;
}

// Counts one record per lane (lanes with `have`; every lane of the warp calls).
//
// One word: a first probe round, and a round of the queue whenever it
// holds a full warp, so that every round has full warps (one record in seven
// needs a second round at half a table; looping until the last lane is done
// took two to three rounds with few lanes each).
template <int W>
__device__ __forceinline__ void count_record(const Table& t, const unsigned long long (&rec)[W], bool have,
                                             unsigned ngroups, unsigned& waiting, unsigned* s_flags) {
    if constexpr (W == 1) {
        const unsigned hsh = leaf_hash(rec[0]);
        probe_round(t, rec[0], have, __umulhi(hsh, ngroups), 0u, hsh, ngroups, waiting, s_flags);
        while (waiting >= 32u) probe_queue(t, ngroups, waiting, s_flags);
    } else {
        int slot = kClaimed;
        if (have) slot = find_slot<W>(t, rec, ngroups);
        if (slot >= 0) tally(t, (unsigned)slot, rec[W - 1]);
        else if (slot != kClaimed) atomicOr(s_flags, slot == kGaveUp ? kLeafTimeout : kLeafFull);
        __syncwarp();
    }
}

// The records still waiting after a leaf's last one.
template <int W>
__device__ __forceinline__ void count_waiting(const Table& t, unsigned ngroups, unsigned& waiting, unsigned* s_flags) {
    if constexpr (W == 1)
        while (waiting) probe_queue(t, ngroups, waiting, s_flags);
}

// Clears a warp's slice [s0, s0 + per) of the table (per a multiple of 4).
template <int W>
__device__ __forceinline__ void clear_slice(const Table& t, unsigned s0, unsigned per) {
    const unsigned lane = threadIdx.x & 31;
    // keys: tails, or (tail, head) pairs; head planes of empty slots are never read
    const unsigned k = t.tail + (W == 2 ? 16 : 8) * s0, l = t.lanes + 4 * s0;
    for (unsigned i = 16 * lane; i < (W == 2 ? 16 : 8) * per; i += 512) sts128_zero(k + i);
    for (unsigned i = 16 * lane; i < 4 * per; i += 512) {
#pragma unroll
        for (unsigned p = 0; p < kLanePlanes; ++p) sts128_zero(l + 4 * p * t.stride + i);
    }
}

// Clears the whole table (all threads of the CTA; cap a multiple of 64).
template <int W>
__device__ __forceinline__ void clear_table(const Table& t, unsigned cap) {
    clear_slice<W>(t, (threadIdx.x >> 5) * (cap / kLeafWarps), cap / kLeafWarps);
}

// Sweeps slots [0, cap): k-mers below min_count are dropped, survivors are
// classified and written (one output reservation per warp), and every slot
// is left clear.  Each warp takes a slice of cap / 16 slots: it lists its
// survivors (four slots per lane and step, so that a slice takes two or three
// steps), writes them with full warps, and clears the slice with 16-byte
// stores.
template <int W>
__device__ __forceinline__ void sweep_table(const Job& j, const Table& t, const LeafInfo& li, unsigned cap,
                                            unsigned& distinct) {
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned plane = 4 * t.stride;
    const unsigned per = cap / kLeafWarps;  // a multiple of 4
    const unsigned s0 = wid * per;
    const unsigned more = j.min_count - 1;  // records besides the one that claimed the slot
    const unsigned mylist = t.list + 2 * s0, before = (1u << lane) - 1u;
    unsigned count = 0;
    for (unsigned b = 0; b < per; b += 128) {
        unsigned occ[4], p0[4], p1[4], p2[4];
        // W = 2: keys are 16 bytes a slot, so neighbouring lanes take neighbouring slots
        if constexpr (W == 2) {
#pragma unroll
            for (unsigned q = 0; q < 4; ++q) {
                const unsigned o = b + 32 * q + lane, s = s0 + o;
                occ[q] = p0[q] = p1[q] = p2[q] = 0u;
                if (o < per) {
                    occ[q] = lds32(t.tail + 16 * s);
                    p0[q] = lds32(t.lanes + 4 * s);
                    p1[q] = lds32(t.lanes + plane + 4 * s);
                    p2[q] = lds32(t.lanes + 2 * plane + 4 * s);
                }
            }
        } else {
            const unsigned o = b + 4 * lane, s = s0 + o;
            uint4 x = make_uint4(0u, 0u, 0u, 0u), y = x, a0 = x, a1 = x, a2 = x;
            if (o < per) {
                x = lds128(t.tail + 8 * s);
                y = lds128(t.tail + 8 * s + 16);
                a0 = lds128(t.lanes + 4 * s);
                a1 = lds128(t.lanes + plane + 4 * s);
                a2 = lds128(t.lanes + 2 * plane + 4 * s);
            }
            occ[0] = x.x; occ[1] = x.z; occ[2] = y.x; occ[3] = y.z;
            p0[0] = a0.x; p0[1] = a0.y; p0[2] = a0.z; p0[3] = a0.w;
            p1[0] = a1.x; p1[1] = a1.y; p1[2] = a1.z; p1[3] = a1.w;
            p2[0] = a2.x; p2[1] = a2.y; p2[2] = a2.z; p2[3] = a2.w;
        }
#pragma unroll
        for (unsigned q = 0; q < 4; ++q) {
            // the five left lanes, two halves at a time (their sum is below 65536: no carry)
            const unsigned h = p0[q] + p1[q] + (p2[q] & 0xFFFFu);
            const bool ok = occ[q] != 0u && (h & 0xFFFFu) + (h >> 16) >= more;
            distinct += occ[q] != 0u ? 1u : 0u;
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok)
                sts16(mylist + 2 * (count + __popc(m & before)), s0 + (W == 2 ? b + 32 * q + lane : b + 4 * lane + q));
            count += __popc(m);
        }
    }
    __syncwarp();
    unsigned long long wbase = 0;
    if (lane == 0 && count) wbase = atomicAdd(j.out_n, (unsigned long long)count);
    wbase = __shfl_sync(0xffffffffu, wbase, 0);
    for (unsigned i = lane; i < count; i += 32) {
        const unsigned s = lds16(mylist + 2 * i);
        const unsigned long long pos = wbase + i;
        const unsigned long long tl = slot_tail<W>(t, s);
        unsigned pl[kLanePlanes];
#pragma unroll
        for (unsigned p = 0; p < kLanePlanes; ++p) pl[p] = lds32(t.lanes + p * plane + 4 * s);
        unsigned long long key[W];
#pragma unroll
        for (int w = 0; w < W - 1; ++w) key[w] = lds64(head_addr<W>(t, w, s));
        if (pos >= j.out_cap) {
            set_status(j, ST_OUT_OVERFLOW);
            continue;
        }
        unsigned nl[4] = {pl[0] & 0xFFFFu, pl[0] >> 16, pl[1] & 0xFFFFu, pl[1] >> 16};
        unsigned nr[4] = {pl[2] >> 16, pl[3] & 0xFFFFu, pl[3] >> 16, pl[4] & 0xFFFFu};
        const unsigned c = 1u + nl[0] + nl[1] + nl[2] + nl[3] + (pl[2] & 0xFFFFu);
        const unsigned code = ((unsigned)tl & 63u) - 1u, fl = ext_left(code), fr = ext_right(code);  // the first record
#pragma unroll
        for (unsigned b = 0; b < 4; ++b) {
            nl[b] += fl == b + 1u ? 1u : 0u;
            nr[b] += fr == b + 1u ? 1u : 0u;
        }
        const unsigned long long z = record_z(j.g, j.pass, j.bucket0 + li.bucket, tl);
        key[W - 1] = z_to_tail<W>(z, key, j.g.bt);
#pragma unroll
        for (int w = 0; w < W; ++w) j.out_keys[pos * W + w] = key[w];
        j.out_count[pos] = c;
        uint4* eo = reinterpret_cast<uint4*>(j.out_ext + pos * 8);
        eo[0] = make_uint4(nl[0], nl[1], nl[2], nl[3]);
        eo[1] = make_uint4(nr[0], nr[1], nr[2], nr[3]);
        reinterpret_cast<uchar2*>(j.out_cls)[pos] = make_uchar2(classify_side(nl, c, j), classify_side(nr, c, j));
    }
    __syncwarp();
    clear_slice<W>(t, s0, per);
}

// A leaf whose keys did not fit its table (and that has fewer than 65 536
// records): counted first as a whole in the whole table, then, if its keys
// still do not fit, in key ranges.  A range (rb, rs) holds the records whose
// next rb z bits below the leaf's bits equal rs; a range that does not fit is
// split in two, down to kMaxSubBits levels, in depth-first order, and a range
// that does not fit at the last level is handed to the HBM recount.  The
// table is clean on entry and on return.  Returns the windows this thread
// counted.
template <int W>
__device__ __forceinline__ unsigned count_in_ranges(const Job& j, const Table& t, const LeafInfo& li, unsigned leaf,
                                                 unsigned* s_flags, unsigned* distinct) {
    const unsigned n = (unsigned)li.n;  // below 65 536
    const unsigned zb = j.g.zl_bits();
    const unsigned free_bits = zb > j.g.p2 ? zb - j.g.p2 : 0u;  // z bits below the leaf's
    const unsigned max_rb = free_bits < kMaxSubBits ? free_bits : kMaxSubBits;
    const unsigned cap = t.stride;
    const unsigned long long* src = li.recs + li.start * W;
    unsigned windows = 0;
    unsigned rb = 0, rs = 0;
    for (;;) {
        const unsigned shift = free_bits - rb, rmask = (1u << rb) - 1u;
        unsigned rwin = 0, waiting = 0;
        for (unsigned i0 = 0; i0 < n; i0 += kLeafThreads) {
            const unsigned i = i0 + threadIdx.x;
            unsigned long long rec[W];
#pragma unroll
            for (int w = 0; w < W; ++w) rec[w] = i < n ? src[(size_t)i * W + w] : 0ull;
            const bool in = i < n && ((unsigned)((rec[W - 1] >> 6) >> shift) & rmask) == rs;
            rwin += in ? 1u : 0u;
            count_record<W>(t, rec, in && !*(volatile unsigned*)s_flags, groups_of<W>(cap), waiting, s_flags);
        }
        count_waiting<W>(t, groups_of<W>(cap), waiting, s_flags);
        __syncthreads();
        const unsigned flags = *(volatile unsigned*)s_flags;
        if (flags == kLeafFull && rb < max_rb) {  // split the range in two
            if (threadIdx.x == 0 && rb == 0) atomicAdd(j.stats + 3, 1ull);
            clear_table<W>(t, cap);
            __syncthreads();
            if (threadIdx.x == 0) *s_flags = 0;
            __syncthreads();
            ++rb;
            rs <<= 1;
            continue;
        }
        if (flags) {
            if (threadIdx.x == 0) {
                if (flags & kLeafTimeout) {
                    set_status(j, ST_TIMEOUT);
                } else {  // exact recount of the range in HBM
                    const unsigned idx = atomicAdd(j.fb_n, 1u);
                    if (idx < j.fb_cap) j.fb_list[idx] = fallback_entry(leaf, rb, rs);
                    else set_status(j, ST_FALLBACK_FULL);
                }
            }
            clear_table<W>(t, cap);
        } else {
            windows += rwin;
            sweep_table<W>(j, t, li, cap, *distinct);
        }
        __syncthreads();
        if (threadIdx.x == 0) *s_flags = 0;
        __syncthreads();
        // next range in depth-first order: climb while this range was a right half
        while (rb > 0 && (rs & 1u)) {
            rs >>= 1;
            --rb;
        }
        if (rb == 0) break;
        ++rs;
    }
    return windows;
}

// Leaves whose keys did not fit their table in leaf_kernel (the split list of
// each analysis), counted in key ranges.  Persistent CTAs over the listed
// leaves of every analysis; each analysis's list is complete when this
// kernel starts.
template <int W>
__global__ void __launch_bounds__(kLeafThreads, 2) leaf_split_kernel(const Job* __restrict__ jobs,
                                                                    const unsigned n_jobs, const unsigned cap_max) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned s_flags;
    const int lane = threadIdx.x & 31;
    Table t;
    t.stride = cap_max;
    t.tail = (unsigned)__cvta_generic_to_shared(smem);
    t.heads = t.tail + 8 * cap_max;
    t.lanes = t.heads + 8 * (W - 1) * cap_max;
    t.list = t.lanes + 4 * kLanePlanes * cap_max;
    t.queue = t.list + 2 * cap_max + (threadIdx.x >> 5) * kQueue * 12;  // 128-byte aligned
    bool init = false;
    for (unsigned ji = 0; ji < n_jobs; ++ji) {
        const Job& j = jobs[ji];
        const unsigned n_split = *(volatile unsigned*)j.split_n;
        if (blockIdx.x >= n_split) continue;
        if (!init) {
            clear_table<W>(t, cap_max);
            if (threadIdx.x == 0) s_flags = 0;
            __syncthreads();
            init = true;
        }
        unsigned long long windows = 0;
        unsigned distinct = 0;
        for (unsigned e = blockIdx.x; e < n_split; e += gridDim.x) {
            const unsigned leaf = j.split_list[e];
            const LeafInfo li = leaf_info(j, leaf);
            windows += count_in_ranges<W>(j, t, li, leaf, &s_flags, &distinct);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            windows += __shfl_xor_sync(0xffffffffu, windows, o);
            distinct += __shfl_xor_sync(0xffffffffu, distinct, o);
        }
        if (lane == 0 && windows) atomicAdd(j.stats + 0, windows);
        if (lane == 0 && distinct) atomicAdd(j.stats + 1, distinct);
    }
}

// Persistent CTAs over the leaves of every analysis of key width W; `leaf_off`
// is the exclusive prefix (n_jobs + 1) of the analyses' leaf counts.
template <int W>
__global__ void __launch_bounds__(kLeafThreads, 2) leaf_kernel(const Job* __restrict__ jobs,
                                                              const unsigned long long* __restrict__ leaf_off,
                                                              const unsigned n_jobs, const unsigned cap_max) {
    constexpr int U = LeafShape<W>::U, B = LeafShape<W>::B;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned s_flags;
    __shared__ Job s_job;        // the current analysis: its fields are read in every phase of every leaf
    __shared__ LeafInfo s_next;  // the next leaf, looked up by one thread while this one is counted
    const int lane = threadIdx.x & 31;
    const unsigned long long total = leaf_off[n_jobs];
    static_assert(sizeof(Job) % 4 == 0, "copied word by word");
    auto take_job = [&](unsigned ji) {
        for (unsigned i = threadIdx.x; i < sizeof(Job) / 4; i += kLeafThreads)
            reinterpret_cast<unsigned*>(&s_job)[i] = reinterpret_cast<const unsigned*>(jobs + ji)[i];
    };

    Table t;
    t.stride = cap_max;
    t.tail = (unsigned)__cvta_generic_to_shared(smem);
    t.heads = t.tail + 8 * cap_max;
    t.lanes = t.heads + 8 * (W - 1) * cap_max;
    t.list = t.lanes + 4 * kLanePlanes * cap_max;
    t.queue = t.list + 2 * cap_max + (threadIdx.x >> 5) * kQueue * 12;  // 128-byte aligned
    clear_table<W>(t, cap_max);
    if (threadIdx.x == 0) s_flags = 0;

    // statistics of the current analysis, added when the analysis changes
    unsigned long long windows = 0;
    unsigned distinct = 0;  // of this thread's slots: far below 2^32
    unsigned stat_job = 0;
    auto flush_stats = [&](unsigned ji) {
        unsigned long long d = distinct;
#pragma unroll
        for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0 && d) atomicAdd(jobs[ji].stats + 1, d);
        if (threadIdx.x == 0 && windows) atomicAdd(jobs[ji].stats + 0, windows);
        windows = 0;
        distinct = 0;
    };

    unsigned long long g = blockIdx.x;
    unsigned ji = 0;
    unsigned leaf = 0;
    LeafInfo li;
    li.ok = false;
    unsigned long long batch[U][W];
    if (g < total) {
        ji = job_of(leaf_off, n_jobs, g);
        leaf = (unsigned)(g - leaf_off[ji]);
        li = leaf_info(jobs[ji], leaf);
        load_batch<W>(li, 0, batch);
        stat_job = ji;
        take_job(ji);
    }
    __syncthreads();

    const Job& j = s_job;
    while (g < total) {
        if (ji != stat_job) {
            flush_stats(stat_job);
            stat_job = ji;
            __syncthreads();  // every thread is done with the previous analysis
            take_job(ji);
            __syncthreads();
        }
        const unsigned long long ng = g + gridDim.x;
        unsigned nji = ji, nleaf = 0;
        if (ng < total) {
            nji = job_of(leaf_off, n_jobs, ng);
            nleaf = (unsigned)(ng - leaf_off[nji]);
        }
        if (!li.ok || li.n >= 65536ull) {
            if (li.ok && threadIdx.x == 0) {  // 16-bit tallies could wrap: exact recount in HBM
                const unsigned idx = atomicAdd(j.fb_n, 1u);
                if (idx < j.fb_cap) j.fb_list[idx] = fallback_entry(leaf, 0, 0); else set_status(j, ST_FALLBACK_FULL);
            }
            g = ng;
            ji = nji;
            leaf = nleaf;
            li.ok = false;
            if (g < total) {
                li = leaf_info(jobs[ji], leaf);
                load_batch<W>(li, 0, batch);
            }
            continue;
        }
        // ---------------------------------------------------------- count
        const unsigned n = (unsigned)li.n;  // below 65 536, as is the ratio (at most 65 536)
        // twice the expected keys and 1024: emptier tables probe less than their
        // sweep costs (256 / 512 / 1280 in place of 1024 at k = 55 with the gate:
        // 1.57 / 1.45 / 1.28 ms)
        const unsigned want = (unsigned)(((unsigned long long)n * j.table_ratio_num) >> 16) + 1024u;
        const unsigned cap = want < cap_max ? ((want + 63u) & ~63u) : cap_max;
        const unsigned ngroups = groups_of<W>(cap);
        if (threadIdx.x == kLeafThreads - 1) {
            LeafInfo x;
            x.ok = false;
            if (ng < total) x = leaf_info(jobs[nji], nleaf);
            s_next = x;
        }
        unsigned waiting = 0;  // records in this warp's queue
        for (unsigned first = 0; first < n; first += B) {
            if (first) load_batch<W>(li, first, batch);
            if (__any_sync(0xffffffffu, *(volatile unsigned*)&s_flags != 0u)) break;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                count_record<W>(t, batch[u], first + u * kLeafThreads + threadIdx.x < n, ngroups, waiting, &s_flags);
            }
        }
        count_waiting<W>(t, ngroups, waiting, &s_flags);
        __syncthreads();
        const unsigned flags = s_flags;
        // the next leaf's first batch loads while this one is swept
        const LeafInfo nli = s_next;
        load_batch<W>(nli, 0, batch);
        if (flags) {
            if (threadIdx.x == 0) {
                if (flags & kLeafTimeout) {
                    set_status(j, ST_TIMEOUT);
                } else {  // keys did not fit: counted again, in key ranges (leaf_split_kernel)
                    const unsigned idx = atomicAdd(j.split_n, 1u);
                    if (idx < j.split_cap) {
                        j.split_list[idx] = leaf;
                    } else {
                        const unsigned f = atomicAdd(j.fb_n, 1u);
                        if (f < j.fb_cap) j.fb_list[f] = fallback_entry(leaf, 0, 0);
                        else set_status(j, ST_FALLBACK_FULL);
                    }
                }
            }
            // every warp has read the flags before thread 0 clears them below: one that
            // came late would sweep a table that is only partly counted
            __syncthreads();
            clear_table<W>(t, cap);  // leave the table clean
        } else {
            if (threadIdx.x == 0) windows += n;
            sweep_table<W>(j, t, li, cap, distinct);  // filter, classify, compact (per warp)
        }
        if (threadIdx.x == 0) s_flags = 0;
        __syncthreads();  // the clean table is reused by the next leaf
        g = ng;
        ji = nji;
        leaf = nleaf;
        li = nli;
    }
    if (blockIdx.x < total) flush_stats(stat_job);
}

template <int W>
static cudaError_t launch_leaf_w(const Job* jobs, const unsigned long long* leaf_off, unsigned n_jobs,
                                 unsigned long long leaves, unsigned cap_max, int num_sms, cudaStream_t s) {
    const size_t smem = leaf_smem_bytes(W, cap_max);
    cudaError_t e = raise_smem_limit((const void*)leaf_kernel<W>, smem);
    if (e != cudaSuccess) return e;
    unsigned long long grid = (unsigned long long)num_sms * 2;
    if (grid > leaves) grid = leaves;
    if (grid == 0) return cudaSuccess;
    leaf_kernel<W><<<(unsigned)grid, kLeafThreads, smem, s>>>(jobs, leaf_off, n_jobs, cap_max);
    return cudaGetLastError();
}

template <int W>
static cudaError_t launch_leaf_split_w(const Job* jobs, unsigned n_jobs, unsigned cap_max, int num_sms,
                                       cudaStream_t s) {
    const size_t smem = leaf_smem_bytes(W, cap_max);
    cudaError_t e =
        raise_smem_limit((const void*)leaf_split_kernel<W>, smem);
    if (e != cudaSuccess) return e;
    if (n_jobs == 0) return cudaSuccess;
    leaf_split_kernel<W><<<(unsigned)num_sms * 2, kLeafThreads, smem, s>>>(jobs, n_jobs, cap_max);
    return cudaGetLastError();
}

cudaError_t launch_leaf_split(unsigned W, const Job* jobs, unsigned n_jobs, unsigned cap_max, int num_sms,
                              cudaStream_t s) {
    switch (W) {
        case 1: return launch_leaf_split_w<1>(jobs, n_jobs, cap_max, num_sms, s);
        case 2: return launch_leaf_split_w<2>(jobs, n_jobs, cap_max, num_sms, s);
        case 3: return launch_leaf_split_w<3>(jobs, n_jobs, cap_max, num_sms, s);
        case 4: return launch_leaf_split_w<4>(jobs, n_jobs, cap_max, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_leaf(unsigned W, const Job* jobs, const unsigned long long* leaf_off, unsigned n_jobs,
                        unsigned long long leaves, unsigned cap_max, int num_sms, cudaStream_t s) {
    switch (W) {
        case 1: return launch_leaf_w<1>(jobs, leaf_off, n_jobs, leaves, cap_max, num_sms, s);
        case 2: return launch_leaf_w<2>(jobs, leaf_off, n_jobs, leaves, cap_max, num_sms, s);
        case 3: return launch_leaf_w<3>(jobs, leaf_off, n_jobs, leaves, cap_max, num_sms, s);
        case 4: return launch_leaf_w<4>(jobs, leaf_off, n_jobs, leaves, cap_max, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kmer
