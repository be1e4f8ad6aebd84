// Survivors in ascending key order (KMER_FLAG_SORTED_OUTPUT).  The k-mer set
// is a set (Sec. II-A use case 1: inserts commute), so its order is free; the
// partitions leave it grouped by the mixed key.  Two sorts: a sample sort
// (below, second half of this file), and a digit-by-digit sort that takes over
// above 2^28 survivors and when thousands of keys begin with the same 64 bits.
//
// Digit by digit (least significant first): 8-bit digits over the 2k key
// bits; each survivor's position is carried along; the counts, tallies and
// classes travel as one 64-byte record per survivor (written while the digits
// are counted) and are gathered through that permutation straight into the
// result arrays, one random record read per survivor.
//
// One kernel per digit (a one-sweep pass): each CTA takes the next tile of
// keys, ranks them by digit within the tile (stable: warps own consecutive
// runs of keys, lanes of one digit are ordered by lane), publishes its
// per-digit counts, and sums the counts of the tiles before it by looking
// back along a per-(tile, digit) status array (decoupled look-back: a tile's
// inclusive prefix, once known, ends the walk of every later tile).  The
// tile is then reordered by digit in shared memory and written out, so each
// digit's keys leave as one contiguous run.  The digit totals of every pass
// come from one histogram kernel over the keys; passes whose digit is the
// same for every key are skipped.
#include <algorithm>
#include <vector>

#include "kernels.h"

namespace kmer {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr unsigned kSortSpinBudget = 1u << 22;  // look-back polls per thread before giving up
constexpr int kLookBack = 8;                     // predecessors read per look-back step

template <int W>
struct SortShape {
    // keys per thread and CTAs per SM (the registers are bounded for it): a
    // pass holds only one word per key in registers, so occupancy is set by
    // the shared-memory tile; measured on 114 M one-word keys, 8 keys at six
    // CTAs per SM ran a pass in 0.86 ms against 1.16 ms for 12 keys at three
    static constexpr int ITEMS = W <= 2 ? 8 : 4;
    static constexpr int MINB = W == 1 ? 6 : 4;
    static constexpr int TILE = kSortThreads * ITEMS;
    static constexpr size_t SMEM = (size_t)TILE * W * 8 + (size_t)TILE * 4;  // reordered keys + positions
};

// Digit `pass` (bits [8 pass, 8 pass + 8) of the key value) of a key: word
// W - 1 - 8 pass / 64, shifted right by 8 pass % 64 (a select, not an indexed
// load, so the key stays in registers).
template <int W>
__device__ __forceinline__ unsigned digit_of(const unsigned long long (&key)[W], unsigned pass) {
    const unsigned wi = W - 1 - (8 * pass) / 64, sh = (8 * pass) % 64;
    unsigned long long v = key[0];
#pragma unroll
    for (int w = 1; w < W; ++w) v = (unsigned)w == wi ? key[w] : v;
    return (unsigned)(v >> sh) & 0xFFu;
}

// A survivor's payload while the keys are sorted, 64 bytes (written whole,
// so no sector is partly written): (count, classes left | right << 8, 0, 0),
// ext[0..3], ext[4..7], zeros.
constexpr int kRecU4 = 4;

// hist[p * 256 + d] = keys whose digit p is d, for p < passes; rec[i] = the
// payload record of survivor i.
template <int W>
__global__ void __launch_bounds__(kSortThreads) sort_digits_kernel(const unsigned long long* __restrict__ keys,
                                                                   const unsigned* __restrict__ count,
                                                                   const unsigned* __restrict__ ext,
                                                                   const unsigned char* __restrict__ cls,
                                                                   unsigned long long n, unsigned passes,
                                                                   unsigned* __restrict__ hist,
                                                                   uint4* __restrict__ rec) {
    extern __shared__ unsigned h[];  // passes * 256
    for (unsigned i = threadIdx.x; i < passes * 256; i += kSortThreads) h[i] = 0;
    __syncthreads();
    for (unsigned long long i = blockIdx.x * (unsigned long long)kSortThreads + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * kSortThreads) {
        unsigned long long key[W];
#pragma unroll
        for (int w = 0; w < W; ++w) key[w] = keys[i * W + w];
        const uchar2 c2 = reinterpret_cast<const uchar2*>(cls)[i];
        const uint4* e = reinterpret_cast<const uint4*>(ext + i * 8);
        uint4* r = rec + i * kRecU4;
        r[0] = make_uint4(count[i], (unsigned)c2.x | (unsigned)c2.y << 8, 0u, 0u);
        r[1] = e[0];
        r[2] = e[1];
        r[3] = make_uint4(0u, 0u, 0u, 0u);
        for (unsigned p = 0; p < passes; ++p) atomicAdd(&h[p * 256 + digit_of<W>(key, p)], 1u);
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < passes * 256; i += kSortThreads)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

__device__ __forceinline__ unsigned long long poll(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void publish(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Exclusive scan of one value per thread over the CTA (256 threads).
__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned* warp_tot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    unsigned before = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w)
        if (w < wid) before += warp_tot[w];
    __syncthreads();
    return before + x - v;
}

// One pass: keys (and positions; identity when isrc is null) from src to dst
// ordered by digit `pass`.  status: tiles * 256 words (stamp << 32 | count),
// stamps 2 s + 1 (the tile's own count) and 2 s + 2 (its inclusive prefix)
// for the s-th pass of this sort; tile_counter: zero before the pass.
// Only the key word that holds the digit is kept in registers while ranking;
// the keys and positions are read again (from L2) when the tile is reordered,
// and the look-back runs after the reorder so its wait overlaps that work.
template <int W>
__global__ void __launch_bounds__(kSortThreads, SortShape<W>::MINB) sort_pass_kernel(
    const unsigned long long* __restrict__ src, const unsigned* __restrict__ isrc, unsigned long long n,
    unsigned pass, unsigned stamp_s, const unsigned* __restrict__ hist, unsigned long long* status,
    unsigned* tile_counter, unsigned long long* __restrict__ dst, unsigned* __restrict__ idst, unsigned* err) {
    constexpr int ITEMS = SortShape<W>::ITEMS, TILE = SortShape<W>::TILE;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long* skeys = reinterpret_cast<unsigned long long*>(smem);
    unsigned* sidx = reinterpret_cast<unsigned*>(smem + (size_t)TILE * W * 8);
    __shared__ unsigned wcnt[kSortWarps][256];  // per warp: keys per digit, then its first rank in the tile
    __shared__ unsigned tstart[256];            // tile-local start of each digit
    __shared__ unsigned long long gbase[256];   // global start of the tile's run of each digit
    __shared__ unsigned warp_tot[kSortWarps];
    __shared__ unsigned s_tile;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned d_me = threadIdx.x;  // the digit this thread looks after in the scans
    const unsigned wi = W - 1 - (8 * pass) / 64, sh = (8 * pass) % 64;  // the digit's word and shift
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_counter, 1u);  // tiles in start order: predecessors run
    for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
    const unsigned long long t = s_tile;
    const unsigned long long t0 = t * TILE;
    const unsigned tile_n = (unsigned)(n - t0 < (unsigned long long)TILE ? n - t0 : TILE);

    // ---- digits and ranks: warp w owns keys [w * 32 * ITEMS, (w + 1) * 32 * ITEMS) of the tile
    unsigned dr[ITEMS];  // digit (9 bits: 256 + lane past the end), then rank << 9 | digit
    const unsigned long long wbase = t0 + (unsigned long long)wid * 32 * ITEMS;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const unsigned long long i = wbase + (unsigned long long)u * 32 + lane;
        dr[u] = i < n ? (unsigned)(src[i * W + wi] >> sh) & 0xFFu : 256u + lane;  // past the end: a digit of its own
    }
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const unsigned d = dr[u];
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned before = __popc(peers & ((1u << lane) - 1u));
        const bool in = d < 256;
        const unsigned run = in ? wcnt[wid][d] : 0u;
        __syncwarp();
        if (in && before == 0) wcnt[wid][d] = run + __popc(peers);
        __syncwarp();
        dr[u] = (run + before) << 9 | d;  // rank among the warp's keys of digit d
    }
    __syncthreads();

    // ---- tile counts per digit: publish them; tile-local starts
    unsigned cnt = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const unsigned c = wcnt[w][d_me];
        wcnt[w][d_me] = cnt;  // warps' first ranks within the digit
        cnt += c;
    }
    const unsigned agg = 2 * stamp_s + 1, inc = 2 * stamp_s + 2;
    unsigned long long* my = status + t * 256 + d_me;
    publish(my, (unsigned long long)(t == 0 ? inc : agg) << 32 | cnt);
    // start of the digit's run among all keys: earlier digits of this pass
    const unsigned dstart = block_excl_scan(__ldg(hist + pass * 256 + d_me), warp_tot);
    tstart[d_me] = block_excl_scan(cnt, warp_tot);
    __syncthreads();

    // ---- reorder the tile by digit in shared memory (keys and positions read again)
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        const unsigned d = dr[u] & 0x1FFu;
        if (d >= 256) continue;
        const unsigned long long i = wbase + (unsigned long long)u * 32 + lane;
        const unsigned lp = tstart[d] + wcnt[wid][d] + (dr[u] >> 9);
#pragma unroll
        for (int w = 0; w < W; ++w) skeys[(size_t)lp * W + w] = src[i * W + w];
        sidx[lp] = isrc ? isrc[i] : (unsigned)i;
    }

    // ---- look-back: keys of this digit in earlier tiles
    unsigned long long prefix = 0;
    if (t > 0) {
        // a window of kLookBack predecessors per step: their words are read
        // together and summed nearest first up to the first inclusive prefix;
        // a predecessor that has not yet published is polled again
        unsigned spins = 0;
        bool gave_up = false;
        long long j = (long long)t - 1;
        for (;;) {
            unsigned long long v[kLookBack];
#pragma unroll
            for (int q = 0; q < kLookBack; ++q)
                v[q] = j - q >= 0 ? poll(status + (unsigned long long)(j - q) * 256 + d_me)
                                  : (unsigned long long)inc << 32;  // before tile 0: an empty prefix
            int q = 0;
            bool done = false;
            for (; q < kLookBack; ++q) {
                const unsigned st = (unsigned)(v[q] >> 32);
                if (st != agg && st != inc) break;
                prefix += v[q] & 0xFFFFFFFFull;
                if (st == inc) {
                    done = true;
                    break;
                }
            }
            if (done) break;
            j -= q;
            if (q < kLookBack) {
                if (++spins > kSortSpinBudget) {
                    gave_up = true;
                    break;
                }
                __nanosleep(32);
            }
        }
        if (gave_up) atomicOr(err, ST_TIMEOUT);
        publish(my, (unsigned long long)inc << 32 | ((prefix + cnt) & 0xFFFFFFFFull));
    }
    gbase[d_me] = (unsigned long long)dstart + prefix;
    __syncthreads();

    // ---- write each digit's run
    for (unsigned j = threadIdx.x; j < tile_n; j += kSortThreads) {
        const unsigned d = (unsigned)(skeys[(size_t)j * W + wi] >> sh) & 0xFFu;
        const unsigned long long g = gbase[d] + (j - tstart[d]);
        if (g >= n) {  // only after a look-back gave up: record it and skip the write
            atomicOr(err, ST_SORT_RANGE);
            continue;
        }
#pragma unroll
        for (int w = 0; w < W; ++w) dst[g * W + w] = skeys[(size_t)j * W + w];
        idst[g] = sidx[j];
    }
}

// The survivors' counts, tallies and classes in the order of `perm`, from
// their payload records (`ext` 16-byte and `cls` 2-byte aligned, as the
// result arrays always are).
__global__ void __launch_bounds__(256) sort_gather_kernel(const unsigned* __restrict__ perm, unsigned long long n,
                                                          const uint4* __restrict__ rec,
                                                          unsigned* __restrict__ count, unsigned* __restrict__ ext,
                                                          unsigned char* __restrict__ cls) {
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += (unsigned long long)gridDim.x * 256) {
        const uint4* r = rec + (unsigned long long)perm[i] * kRecU4;
        const uint4 a = r[0], e0 = r[1], e1 = r[2];
        count[i] = a.x;
        uint4* eo = reinterpret_cast<uint4*>(ext + i * 8);
        eo[0] = e0;
        eo[1] = e1;
        reinterpret_cast<uchar2*>(cls)[i] = make_uchar2((unsigned char)(a.y & 0xFFu), (unsigned char)(a.y >> 8));
    }
}

// ------------------------------------------------------------------------
// Sample sort: the keys are split by value into buckets of about a thousand
// (one level of splitters, or two), and one CTA sorts each bucket in shared
// memory and writes its survivors' keys, counts, tallies and classes where
// they belong.  What moves between the steps is a survivor's position and the
// first 64 bits of its key (12 bytes for any k), so the passes over memory do
// not grow with k; the digit-by-digit sort makes 2k/8 passes over positions
// and whole keys.  Splitters come from the keys themselves, because canonical
// k-mers are anything but uniform (half the density of AAA... at CCC...,
// clusters of a deep k-mer's error variants).  A bucket's exact place is known
// before anything moves (a count pass), so no slack is kept and each bucket is
// sorted into its final range.
//
// Whole sort, against digit by digit: 67 M one-word survivors 9.66 -> 3.96 ms
// (payload records and counts 0.98, two scatters 0.81, level-2 count and
// splitters 0.25, buckets 1.93: 90 bytes a survivor asked for, 101 moved, as a
// random 32-byte record costs more than its sector); 8 M four-word survivors 6.25 -> 0.82 ms; 100 k
// survivors, k = 21 to 99, 78-250 -> 45-60 us (launches).
constexpr int kSplitThreads = 512;
constexpr int kPickThreads = 1024;
constexpr unsigned kMaxFan = 512;          // buckets of one splitting step
constexpr unsigned kSplitTile = 4096;      // elements per tile of a scatter
constexpr unsigned kCountTile = 8192;      // elements per tile of a level-2 count
constexpr unsigned kSplitItems = kSplitTile / kSplitThreads;
constexpr unsigned kBucketItems = 6;       // elements per thread of a bucket's CTA
constexpr unsigned kBucketCap = kBucketItems * kSplitThreads;  // elements a bucket may have
constexpr unsigned kBucketMean = 1152;     // mean bucket: 3/8 of the capacity
constexpr unsigned kMaxSamples = 16384;
constexpr unsigned long long kSampleSortMax = 1ull << 28;  // survivors: kMaxFan^2 buckets near their mean size

// First 64 bits of key i, left-aligned (hb = bits of word 0); W = 0: `a`
// holds them.  They order one-word keys completely.
template <int W>
__device__ __forceinline__ unsigned long long prefix_at(const unsigned long long* a, unsigned long long i,
                                                        unsigned hb) {
    if constexpr (W == 0) return a[i];
    else if constexpr (W == 1) return a[i] << (64 - hb);
    else return (a[i * W] << (64 - hb)) | (a[i * W + 1] >> hb);
}

// Group g of a step: elements [start[g], start[g + 1]), or all n (start null).
__device__ __forceinline__ void group_range(const unsigned* start, unsigned g, unsigned n, unsigned& a, unsigned& cnt) {
    a = start ? start[g] : 0u;
    cnt = (start ? start[g + 1] : n) - a;
}

// Buckets of a group of `cnt` elements: `mean` elements each, at most `stride` buckets.
__host__ __device__ inline unsigned buckets_for(unsigned cnt, unsigned mean, unsigned stride) {
    const unsigned b = cnt / mean + (cnt % mean ? 1u : 0u);
    return b < 1u ? 1u : (b > stride ? stride : b);
}

// Exclusive scan of one value per thread over a CTA of NT threads (all call).
template <unsigned NT>
__device__ __forceinline__ unsigned block_scan(unsigned v, unsigned* warp_tot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    unsigned t = lane < (int)(NT / 32) ? warp_tot[lane] : 0u;
#pragma unroll
    for (unsigned o = 1; o < NT / 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= (int)o) t += y;
    }
    const unsigned before = __shfl_sync(0xffffffffu, t, wid ? wid - 1 : 0);
    __syncthreads();
    return (wid ? before : 0u) + x - v;
}

// Splitters of a group and the table that finds an element's bucket: prefixes
// from `lo` on are cut into kLut ranges of 2^shift; first[b] = splitters in
// ranges before b, so the bucket is found among the few splitters of one range.
constexpr unsigned kLut = 2048;
struct SplitTable {
    unsigned long long lo;
    unsigned shift, pad;
    unsigned long long spl[kMaxFan];  // nb - 1 splitters, ascending
    unsigned short first[kLut + 8];
};

__device__ __forceinline__ unsigned range_of(unsigned long long p, unsigned long long lo, unsigned shift) {
    const unsigned long long r = (p > lo ? p - lo : 0ull) >> shift;
    return r < kLut ? (unsigned)r : kLut - 1;
}

// How many splitters are <= p (a binary search over those of p's range).
__device__ __forceinline__ unsigned bucket_of(const SplitTable& t, unsigned long long p) {
    const unsigned r = range_of(p, t.lo, t.shift);
    unsigned l = t.first[r], h = t.first[r + 1];
    while (l < h) {
        const unsigned mid = (l + h) >> 1;
        if (t.spl[mid] <= p) l = mid + 1; else h = mid;
    }
    return l;
}

// The parts of a table that a group with nb buckets uses, into shared memory (all threads of the CTA).
__device__ __forceinline__ void load_table(SplitTable& d, const SplitTable& t, unsigned nb) {
    if (threadIdx.x == 0) {
        d.lo = t.lo;
        d.shift = t.shift;
    }
    for (unsigned i = threadIdx.x; i + 1 < nb; i += blockDim.x) d.spl[i] = t.spl[i];
    const uint4* f = reinterpret_cast<const uint4*>(t.first);
    for (unsigned i = threadIdx.x; i < (kLut + 8) / 8; i += blockDim.x) reinterpret_cast<uint4*>(d.first)[i] = f[i];
}

// Smallest and largest of the threads' values over the CTA (s: two words).
__device__ __forceinline__ void block_min_max(unsigned long long& lo, unsigned long long& hi, unsigned long long* s) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, lo, o), y = __shfl_xor_sync(0xffffffffu, hi, o);
        lo = x < lo ? x : lo;
        hi = y > hi ? y : hi;
    }
    if (threadIdx.x == 0) {
        s[0] = ~0ull;
        s[1] = 0ull;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&s[0], lo);
        atomicMax(&s[1], hi);
    }
    __syncthreads();
    lo = s[0];
    hi = s[1];
}

// Shift that leaves at most 11 bits of a span: 2048 ranges.
__device__ __forceinline__ unsigned span_shift(unsigned long long span) {
    const int sh = 64 - __clzll((long long)span) - 11;
    return sh > 0 ? (unsigned)sh : 0u;
}

// Exclusive scan of kLut counters in shared memory by a CTA of NT threads;
// returns whether a counter is above `crowd`.
template <unsigned NT>
__device__ __forceinline__ bool scan_ranges(unsigned* bin, unsigned total, unsigned* warp_tot, unsigned crowd) {
    constexpr unsigned PER = kLut / NT;
    static_assert(PER * NT == kLut, "whole runs");
    unsigned v[PER], sum = 0;
    bool far = false;
#pragma unroll
    for (unsigned i = 0; i < PER; ++i) {
        v[i] = bin[threadIdx.x * PER + i];
        sum += v[i];
        far = far || v[i] > crowd;
    }
    unsigned run = block_scan<NT>(sum, warp_tot);
#pragma unroll
    for (unsigned i = 0; i < PER; ++i) {
        bin[threadIdx.x * PER + i] = run;
        run += v[i];
    }
    if (threadIdx.x == 0) bin[kLut] = total;
    return __syncthreads_or(far);
}

// Elements 0 .. m - 1 of a CTA's shared memory into ascending order by a bitonic
// network whose comparators all point up (the places past m stand for elements
// larger than any and never move): log^2 steps whatever the keys.  The
// counting within a range takes as many steps as the range has elements, and
// keys alike in their first bits (error variants of a deep k-mer, amplicons)
// crowd one range, so a CTA with more than crowd_of elements in some range takes
// this way.  4 M survivors in clusters of 10 / 50 / 400 that begin with the same
// 32 bases (16 at k = 31), ms by counting -> as chosen here; random ones; the
// sort by digits:
//   k = 31  0.31 / 0.39 / 1.11 -> 0.31 / 0.39 / 0.53;  0.29;  0.6
//   k = 55  0.61 / 1.32 / 6.49 -> 0.61 / 0.69 / 0.75;  0.38;  1.0
//   k = 99  0.74 / 1.56 / 7.38 -> 0.72 / 0.75 / 0.81;  0.44;  3.1
// The lines lie where the two meet: when counting, equal prefixes of two words
// and more are compared by whole keys in global memory.
template <int W>
__device__ __forceinline__ constexpr unsigned crowd_of() { return W >= 2 ? 32 : 128; }
template <unsigned NT, class Less, class Swap>
__device__ __forceinline__ void sort_crowded(unsigned m, Less less, Swap swap) {
    for (unsigned size = 2; size < 2 * m; size <<= 1) {
        for (unsigned stride = size >> 1; stride; stride >>= 1) {
            for (unsigned t = threadIdx.x;; t += NT) {
                const unsigned low = t & (stride - 1), i = (t - low) << 1 | low;  // bit `stride` clear
                if (i >= m) break;
                const unsigned j = stride == size >> 1 ? i ^ (size - 1) : i | stride;
                if (j < m && less(j, i)) swap(i, j);
            }
            __syncthreads();
        }
    }
}

// One CTA per group: `over` samples per bucket, ordered in shared memory (as
// sort_buckets_kernel orders a bucket); every over-th is a splitter.
template <int W>
__global__ void __launch_bounds__(kPickThreads) split_pick_kernel(const unsigned long long* __restrict__ src,
                                                                  const unsigned* __restrict__ start, unsigned n,
                                                                  unsigned hb, unsigned mean, unsigned over,
                                                                  unsigned stride, SplitTable* __restrict__ tables) {
    constexpr unsigned ITEMS = kMaxSamples / kPickThreads;
    extern __shared__ unsigned long long smp[];
    __shared__ unsigned bin[kLut + 1];
    __shared__ unsigned long long mm[2];
    __shared__ unsigned warp_tot[32];
    const unsigned g = blockIdx.x;
    SplitTable& t = tables[g];
    unsigned a, cnt;
    group_range(start, g, n, a, cnt);
    const unsigned nb = buckets_for(cnt, mean, stride), S = nb > 1 ? nb * over : 0u;
    for (unsigned i = threadIdx.x; i <= kLut; i += kPickThreads) bin[i] = 0;
    unsigned long long v[ITEMS], lo = ~0ull, hi = 0ull;
    unsigned br[ITEMS];
    // evenly spaced places, moved by a hash within their stretch
#pragma unroll
    for (unsigned u = 0; u < ITEMS; ++u) {
        const unsigned i = u * kPickThreads + threadIdx.x;
        v[u] = 0;
        br[u] = 0;
        if (i < S) {
            const unsigned j = (i * 2654435761u + g * 40503u) >> 16;
            const unsigned long long at = (((unsigned long long)i << 16 | j) * cnt) / ((unsigned long long)S << 16);
            v[u] = prefix_at<W>(src, a + at, hb);
            lo = v[u] < lo ? v[u] : lo;
            hi = v[u] > hi ? v[u] : hi;
        }
    }
    block_min_max(lo, hi, mm);
    const unsigned shift = S ? span_shift(hi - lo) : 0u;
#pragma unroll
    for (unsigned u = 0; u < ITEMS; ++u)
        if (u * kPickThreads + threadIdx.x < S) {
            const unsigned b = range_of(v[u], lo, shift);
            br[u] = b | atomicAdd(&bin[b], 1u) << 16;
        }
    __syncthreads();
    const bool crowded = scan_ranges<kPickThreads>(bin, S, warp_tot, crowd_of<1>());
#pragma unroll
    for (unsigned u = 0; u < ITEMS; ++u)
        if (u * kPickThreads + threadIdx.x < S) smp[bin[br[u] & 0xFFFFu] + (br[u] >> 16)] = v[u];
    __syncthreads();
    if (crowded) {
        sort_crowded<kPickThreads>(
            S, [&](unsigned x, unsigned y) { return smp[x] < smp[y]; },
            [&](unsigned x, unsigned y) {
                const unsigned long long a = smp[x];
                smp[x] = smp[y];
                smp[y] = a;
            });
        for (unsigned i = threadIdx.x; i + 1 < nb; i += kPickThreads) t.spl[i] = smp[(i + 1) * over];
    } else {
#pragma unroll
        for (unsigned u = 0; u < ITEMS; ++u)
            if (u * kPickThreads + threadIdx.x < S) {
                const unsigned b = br[u] & 0xFFFFu, b0 = bin[b], b1 = bin[b + 1], me = b0 + (br[u] >> 16);
                unsigned f = b0;
                for (unsigned j = b0; j < b1; ++j) f += smp[j] < v[u] || (smp[j] == v[u] && j < me) ? 1u : 0u;
                if (f % over == 0 && f) t.spl[f / over - 1] = v[u];
            }
    }
    // splitters in ranges before r: those of rank over, 2 over, ... below bin[r]
    for (unsigned r = threadIdx.x; r <= kLut; r += kPickThreads)
        t.first[r] = (unsigned short)(bin[r] ? (bin[r] - 1) / over : 0u);
    if (threadIdx.x == 0) {
        t.lo = S ? lo : 0ull;
        t.shift = shift;
    }
}
// A survivor's payload while the keys are sorted, 32 bytes (one memory
// sector): count, classes (left | right << 8), tallies as 16 bits each.  A
// survivor with a tally past 16 bits (its count is at least 65536, so there are
// at most windows / 65536) sets bit 31 of the classes' word and keeps its
// tallies in the wide list.
constexpr unsigned kWide = 0x80000000u;
constexpr int kSlimU4 = 2;

// Level 1: the bucket of every key, the buckets' sizes, and on the way the
// payload records and (two words and more) the prefixes and a copy of the keys.
template <int W>
__global__ void __launch_bounds__(kSplitThreads) sort_count1_kernel(
    const unsigned long long* __restrict__ keys, const unsigned* __restrict__ count, const unsigned* __restrict__ ext,
    const unsigned char* __restrict__ cls, unsigned n, unsigned hb, const SplitTable* __restrict__ table,
    unsigned nb, unsigned short* __restrict__ ids, unsigned long long* __restrict__ prefix,
    unsigned long long* __restrict__ kcopy, uint4* __restrict__ rec, uint4* __restrict__ wide,
    unsigned* __restrict__ wide_n, unsigned wide_cap, unsigned* __restrict__ size, unsigned* err) {
    __shared__ __align__(16) SplitTable t;
    __shared__ unsigned h[kMaxFan];
    if (nb > 1) load_table(t, *table, nb);
    h[threadIdx.x] = 0;
    __syncthreads();
    for (unsigned long long i = blockIdx.x * (unsigned long long)kSplitThreads + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * kSplitThreads) {
        const unsigned long long p = prefix_at<W>(keys, i, hb);
        const uchar2 c2 = reinterpret_cast<const uchar2*>(cls)[i];
        const uint4* e = reinterpret_cast<const uint4*>(ext + i * 8);
        const uint4 l = e[0], r = e[1];
        unsigned c = (unsigned)c2.x | (unsigned)c2.y << 8;
        uint2 ls = make_uint2(l.x | l.y << 16, l.z | l.w << 16), rs = make_uint2(r.x | r.y << 16, r.z | r.w << 16);
        if ((l.x | l.y | l.z | l.w | r.x | r.y | r.z | r.w) >> 16) {
            const unsigned at = atomicAdd(wide_n, 1u);
            if (at < wide_cap) {
                wide[2 * (size_t)at] = l;
                wide[2 * (size_t)at + 1] = r;
            } else {
                atomicOr(err, ST_SORT_RANGE);  // cannot happen: the counts add up to the windows
            }
            c |= kWide;
            ls.x = at;
        }
        uint4* o = rec + i * kSlimU4;
        o[0] = make_uint4(count[i], c, ls.x, ls.y);
        o[1] = make_uint4(rs.x, rs.y, 0u, 0u);
        if constexpr (W >= 2) {
            if (prefix) prefix[i] = p;
#pragma unroll
            for (int w = 0; w < W; ++w) kcopy[i * W + w] = keys[i * W + w];
        }
        if (nb > 1) {
            const unsigned b = bucket_of(t, p);
            ids[i] = (unsigned short)b;
            atomicAdd(&h[b], 1u);
        }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < nb; i += kSplitThreads)
        if (h[i] && nb > 1) atomicAdd(&size[i], h[i]);
}

// Tiles of a step before each group (tp: groups + 1 entries in shared memory), tile elements each.
__device__ __forceinline__ void tile_prefix(const unsigned* start, unsigned groups, unsigned n, unsigned tile,
                                            unsigned* tp, unsigned* warp_tot) {
    unsigned a = 0, cnt = 0, tiles = 0;
    if (threadIdx.x < groups) {
        group_range(start, threadIdx.x, n, a, cnt);
        tiles = cnt / tile + (cnt % tile ? 1u : 0u);
    }
    const unsigned ex = block_scan<kSplitThreads>(tiles, warp_tot);
    if (threadIdx.x < groups) tp[threadIdx.x] = ex;
    if (threadIdx.x == groups - 1) tp[groups] = ex + tiles;
    __syncthreads();
}

__device__ __forceinline__ unsigned tile_group(const unsigned* tp, unsigned groups, unsigned t) {
    unsigned lo = 0, hi = groups;
    while (hi - lo > 1) {
        const unsigned mid = (lo + hi) >> 1;
        if (tp[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// Level 2: the bucket of every element within its group, and the buckets' sizes.
__global__ void __launch_bounds__(kSplitThreads) sort_count2_kernel(const unsigned long long* __restrict__ prefix,
                                                                    const unsigned* __restrict__ start, unsigned groups,
                                                                    const SplitTable* __restrict__ tables,
                                                                    unsigned mean, unsigned stride,
                                                                    unsigned short* __restrict__ ids,
                                                                    unsigned* __restrict__ size) {
    __shared__ __align__(16) SplitTable tab;
    __shared__ unsigned h[kMaxFan];
    __shared__ unsigned tp[kMaxFan + 1];
    __shared__ unsigned warp_tot[kSplitThreads / 32];
    tile_prefix(start, groups, 0u, kCountTile, tp, warp_tot);
    const unsigned all = tp[groups];
    h[threadIdx.x] = 0;
    for (unsigned t = blockIdx.x; t < all; t += gridDim.x) {
        const unsigned g = tile_group(tp, groups, t);
        unsigned a, cnt;
        group_range(start, g, 0u, a, cnt);
        const unsigned i0 = (t - tp[g]) * kCountTile, m = cnt - i0 < kCountTile ? cnt - i0 : kCountTile;
        load_table(tab, tables[g], buckets_for(cnt, mean, stride));
        __syncthreads();
        const size_t at = (size_t)a + i0;
#pragma unroll 4
        for (unsigned i = threadIdx.x; i < m; i += kSplitThreads) {
            const unsigned b = bucket_of(tab, prefix[at + i]);
            ids[at + i] = (unsigned short)b;
            atomicAdd(&h[b], 1u);
        }
        __syncthreads();
        if (h[threadIdx.x]) {
            atomicAdd(&size[(size_t)g * stride + threadIdx.x], h[threadIdx.x]);
            h[threadIdx.x] = 0;
        }
        // the next tile's table is written after every thread's search (barrier above)
    }
}

// One CTA per group: where each of its buckets starts (bstart: groups * stride
// + 1 entries when there is one group or the buckets of every group are
// consecutive; cursor: a copy that the scatter advances).  A bucket larger
// than `cap` sets ST_SORT_SPLIT: the caller then sorts another way.
__global__ void __launch_bounds__(kSplitThreads) sort_starts_kernel(const unsigned* __restrict__ size,
                                                                    const unsigned* __restrict__ start, unsigned n,
                                                                    unsigned stride, unsigned cap,
                                                                    unsigned* __restrict__ bstart,
                                                                    unsigned* __restrict__ cursor, unsigned* err) {
    __shared__ unsigned warp_tot[kSplitThreads / 32];
    unsigned a, cnt;
    group_range(start, blockIdx.x, n, a, cnt);
    const unsigned v = threadIdx.x < stride ? size[(size_t)blockIdx.x * stride + threadIdx.x] : 0u;
    const unsigned at = a + block_scan<kSplitThreads>(v, warp_tot);
    if (threadIdx.x < stride) {
        bstart[(size_t)blockIdx.x * stride + threadIdx.x] = at;
        cursor[(size_t)blockIdx.x * stride + threadIdx.x] = at;
    }
    if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) bstart[(size_t)gridDim.x * stride] = a + cnt;
    if (v > cap) atomicOr(err, ST_SORT_SPLIT);
}

// Moves the elements of every group to their buckets: tiles are put in bucket
// order in shared memory and leave as one run per bucket (their order within
// a bucket is free: the last step sorts it).  pos null: identity.
template <int W>
__global__ void __launch_bounds__(kSplitThreads, 3) sort_scatter_kernel(
    const unsigned long long* __restrict__ src, const unsigned* __restrict__ pos, const unsigned short* __restrict__ ids,
    const unsigned* __restrict__ start, unsigned groups, unsigned n, unsigned hb, unsigned stride,
    unsigned* __restrict__ cursor, unsigned long long* __restrict__ dst, unsigned* __restrict__ dpos) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long* sp = reinterpret_cast<unsigned long long*>(smem);
    unsigned* si = reinterpret_cast<unsigned*>(sp + kSplitTile);
    unsigned short* sb = reinterpret_cast<unsigned short*>(si + kSplitTile);
    __shared__ unsigned h[kMaxFan], lbase[kMaxFan], wbase[kMaxFan];
    __shared__ unsigned tp[kMaxFan + 1];
    __shared__ unsigned warp_tot[kSplitThreads / 32];
    tile_prefix(start, groups, n, kSplitTile, tp, warp_tot);
    const unsigned all = tp[groups];
    h[threadIdx.x] = 0;
    __syncthreads();
    for (unsigned t = blockIdx.x; t < all; t += gridDim.x) {
        const unsigned g = tile_group(tp, groups, t);
        unsigned a, cnt;
        group_range(start, g, n, a, cnt);
        const unsigned i0 = (t - tp[g]) * kSplitTile, m = cnt - i0 < kSplitTile ? cnt - i0 : kSplitTile;
        const size_t at = (size_t)a + i0;
        unsigned long long p[kSplitItems];
        unsigned q[kSplitItems], br[kSplitItems];
#pragma unroll
        for (unsigned u = 0; u < kSplitItems; ++u) {
            const unsigned i = u * kSplitThreads + threadIdx.x;
            br[u] = 0xFFFFFFFFu;
            if (i < m) {
                br[u] = ids[at + i];
                p[u] = prefix_at<W>(src, at + i, hb);
                q[u] = pos ? pos[at + i] : (unsigned)(at + i);
            }
        }
#pragma unroll
        for (unsigned u = 0; u < kSplitItems; ++u)
            if (br[u] != 0xFFFFFFFFu) br[u] |= atomicAdd(&h[br[u]], 1u) << 16;  // rank within the tile's bucket
        __syncthreads();
        const unsigned c = h[threadIdx.x];
        const unsigned lb = block_scan<kSplitThreads>(c, warp_tot);
        lbase[threadIdx.x] = lb;
        wbase[threadIdx.x] = c ? atomicAdd(&cursor[(size_t)g * stride + threadIdx.x], c) - lb : 0u;
        h[threadIdx.x] = 0;
        __syncthreads();
#pragma unroll
        for (unsigned u = 0; u < kSplitItems; ++u)
            if (br[u] != 0xFFFFFFFFu) {
                const unsigned b = br[u] & 0xFFFFu, at2 = lbase[b] + (br[u] >> 16);
                sp[at2] = p[u];
                si[at2] = q[u];
                sb[at2] = (unsigned short)b;
            }
        __syncthreads();
#pragma unroll
        for (unsigned u = 0; u < kSplitItems; ++u) {
            const unsigned i = u * kSplitThreads + threadIdx.x;
            if (i < m) {
                const size_t to = wbase[sb[i]] + i;
                dst[to] = sp[i];
                dpos[to] = si[i];
            }
        }
        __syncthreads();
    }
}

// Survivor x before y by the words after their first 64 bits, which are equal.
template <int W>
__device__ __forceinline__ bool tail_less(const unsigned long long* __restrict__ keys, unsigned x, unsigned y) {
    const unsigned long long *a = keys + (size_t)x * W, *b = keys + (size_t)y * W;
#pragma unroll
    for (int w = 1; w < W; ++w)
        if (a[w] != b[w]) return a[w] < b[w];
    return false;
}

// A bucket with a crowded range (not inlined: its registers would cost the
// ordinary buckets theirs).  `more` (the ranges' counters, no longer used) holds
// 32 bits after the first 64 of a key where the bucket's elements have room
// there, so that most comparisons of alike keys stay in shared memory.
template <int W>
__device__ __noinline__ void sort_bucket_crowded(unsigned long long* sp, unsigned* si, unsigned* more, unsigned m,
                                                 unsigned hb, const unsigned long long* __restrict__ kcopy) {
    const bool wide = W >= 2 && m <= kLut;
    if constexpr (W >= 2) {
        if (wide)
            for (unsigned i = threadIdx.x; i < m; i += kSplitThreads) {
                const unsigned long long* a = kcopy + (size_t)si[i] * W;
                unsigned long long x = a[1] << (64 - hb);
                if constexpr (W >= 3) x |= a[2] >> hb;
                more[i] = (unsigned)(x >> 32);
            }
        __syncthreads();
    }
    sort_crowded<kSplitThreads>(
        m,
        [&](unsigned x, unsigned y) {
            const unsigned long long a = sp[x], b = sp[y];
            if (W == 1 || a != b) return a < b;
            if (wide && more[x] != more[y]) return more[x] < more[y];
            return tail_less<W>(kcopy, si[x], si[y]);
        },
        [&](unsigned x, unsigned y) {
            const unsigned long long a = sp[x];
            const unsigned c = si[x];
            sp[x] = sp[y];
            si[x] = si[y];
            sp[y] = a;
            si[y] = c;
            if (wide) {
                const unsigned d = more[x];
                more[x] = more[y];
                more[y] = d;
            }
        });
}

// One CTA per bucket.  The elements are spread over kLut ranges of the
// bucket's span of prefixes (about one element a range) and ordered within
// their range by counting the smaller ones (a bucket with a crowded range:
// sort_crowded); equal prefixes (two words and more) are ordered by their whole
// keys.  The survivors are then written in
// order: the key (from the prefix, or from the copy of the keys) and the
// payload record, one random 32-byte read each.  src null: the one bucket of
// all n keys.
template <int W>
__global__ void __launch_bounds__(kSplitThreads, 3) sort_buckets_kernel(
    const unsigned long long* __restrict__ src, const unsigned* __restrict__ pos, const unsigned* __restrict__ bstart,
    unsigned n, unsigned hb, const unsigned long long* __restrict__ kcopy, const uint4* __restrict__ rec,
    const uint4* __restrict__ wide, unsigned wide_cap, const unsigned* __restrict__ err,
    unsigned long long* keys, unsigned* __restrict__ count, unsigned* __restrict__ ext, unsigned char* __restrict__ cls) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long* sp = reinterpret_cast<unsigned long long*>(smem);
    unsigned* si = reinterpret_cast<unsigned*>(sp + kBucketCap);
    unsigned* bin = si + kBucketCap;  // kLut + 1: counts, then starts
    __shared__ unsigned long long mm[2];
    __shared__ unsigned warp_tot[kSplitThreads / 32];
    const unsigned a = bstart ? bstart[blockIdx.x] : 0u, m = (bstart ? bstart[blockIdx.x + 1] : n) - a;
    // an oversized bucket somewhere: nothing is written, the caller sorts another way
    if (m == 0 || m > kBucketCap || (*err & ST_SORT_SPLIT)) return;
    for (unsigned i = threadIdx.x; i < kLut; i += kSplitThreads) bin[i] = 0;
    unsigned long long p[kBucketItems];
    unsigned q[kBucketItems], br[kBucketItems];
    unsigned long long lo = ~0ull, hi = 0ull;
#pragma unroll
    for (unsigned u = 0; u < kBucketItems; ++u) {
        const unsigned i = u * kSplitThreads + threadIdx.x;
        p[u] = 0;
        q[u] = 0;
        if (i < m) {
            p[u] = src ? src[(size_t)a + i] : prefix_at<W>(kcopy ? kcopy : keys, i, hb);
            q[u] = src ? pos[(size_t)a + i] : i;
            lo = p[u] < lo ? p[u] : lo;
            hi = p[u] > hi ? p[u] : hi;
        }
    }
    block_min_max(lo, hi, mm);
    const unsigned shift = span_shift(hi - lo);
#pragma unroll
    for (unsigned u = 0; u < kBucketItems; ++u)
        if (u * kSplitThreads + threadIdx.x < m) {
            const unsigned b = (unsigned)((p[u] - lo) >> shift);
            br[u] = b | atomicAdd(&bin[b], 1u) << 16;
        }
    __syncthreads();
    const bool crowded = scan_ranges<kSplitThreads>(bin, m, warp_tot, crowd_of<W>());
#pragma unroll
    for (unsigned u = 0; u < kBucketItems; ++u)
        if (u * kSplitThreads + threadIdx.x < m) {
            const unsigned at = bin[br[u] & 0xFFFFu] + (br[u] >> 16);
            sp[at] = p[u];
            if (W >= 2 || crowded) si[at] = q[u];
        }
    __syncthreads();
    if (crowded) {
        sort_bucket_crowded<W>(sp, si, bin, m, hb, kcopy);
    } else {
#pragma unroll
        for (unsigned u = 0; u < kBucketItems; ++u)
            if (u * kSplitThreads + threadIdx.x < m) {
                const unsigned b = br[u] & 0xFFFFu, b0 = bin[b], b1 = bin[b + 1], me = b0 + (br[u] >> 16);
                unsigned f = b0;
                if (b1 - b0 > 1)
                    for (unsigned j = b0; j < b1; ++j) {
                        const unsigned long long o = sp[j];
                        bool less = o < p[u];
                        if (W >= 2 && o == p[u] && j != me) {  // whole keys (their first 64 bits are equal)
                            const unsigned long long *x = kcopy + (size_t)si[j] * W, *y = kcopy + (size_t)q[u] * W;
#pragma unroll
                            for (int w = 1; w < W; ++w)
                                if (x[w] != y[w]) {
                                    less = x[w] < y[w];
                                    break;
                                }
                        }
                        f += less ? 1u : 0u;
                    }
                br[u] = f;
            }
        __syncthreads();
#pragma unroll
        for (unsigned u = 0; u < kBucketItems; ++u)
            if (u * kSplitThreads + threadIdx.x < m) {
                sp[br[u]] = p[u];
                si[br[u]] = q[u];
            }
        __syncthreads();
    }
#pragma unroll
    for (unsigned u = 0; u < kBucketItems; ++u) {
        const unsigned i = u * kSplitThreads + threadIdx.x;
        if (i >= m) break;
        const size_t to = (size_t)a + i;
        const unsigned from = si[i];
        const uint4 x = rec[(size_t)from * kSlimU4], y = rec[(size_t)from * kSlimU4 + 1];
        if constexpr (W == 1) {
            keys[to] = sp[i] >> (64 - hb);
        } else {
#pragma unroll
            for (int w = 0; w < W; ++w) keys[to * W + w] = kcopy[(size_t)from * W + w];
        }
        count[to] = x.x;
        uint4 l = make_uint4(x.z & 0xFFFFu, x.z >> 16, x.w & 0xFFFFu, x.w >> 16);
        uint4 r = make_uint4(y.x & 0xFFFFu, y.x >> 16, y.y & 0xFFFFu, y.y >> 16);
        if ((x.y & kWide) && x.z < wide_cap) {
            l = wide[2 * (size_t)x.z];
            r = wide[2 * (size_t)x.z + 1];
        }
        uint4* eo = reinterpret_cast<uint4*>(ext + to * 8);
        eo[0] = l;
        eo[1] = r;
        reinterpret_cast<uchar2*>(cls)[to] = make_uchar2((unsigned char)(x.y & 0xFFu), (unsigned char)(x.y >> 8 & 0xFFu));
    }
}

// Splitting of n survivors: no splitting up to one bucket's capacity, one
// level while its mean bucket allows, else two.
struct SplitPlan {
    unsigned levels, mean, fan1, over1, fan2;
};
static SplitPlan split_plan(unsigned long long n, int num_sms) {
    SplitPlan p{};
    p.mean = kBucketMean;
    if (n <= 1024) return p;  // one bucket: three more launches would cost more than its one CTA takes
    if (n <= (unsigned long long)kMaxFan * kBucketMean) {
        // one level; small inputs take smaller buckets, about two per SM
        const unsigned long long m = n / (2ull * num_sms);
        p.mean = (unsigned)(m < 256 ? 256 : (m > kBucketMean ? kBucketMean : m));
        p.levels = 1;
        p.fan1 = buckets_for((unsigned)n, p.mean, kMaxFan);
        // a bucket of `over` samples varies by 1 / sqrt(over): past the capacity about once in 10^9 buckets
        p.over1 = p.mean <= kBucketCap / 4 ? 16 : 32;
        return p;
    }
    p.levels = 2;
    const unsigned long long b = n / kBucketMean;
    p.fan1 = 1;
    while ((unsigned long long)p.fan1 * p.fan1 < b && p.fan1 < kMaxFan) ++p.fan1;
    p.over1 = 32;
    // level-1 buckets vary by a sixth (32 samples each): room for half as much again
    const unsigned long long f = b / p.fan1 * 3 / 2 + 2;
    p.fan2 = (unsigned)(f > kMaxFan ? kMaxFan : f);
    return p;
}

static size_t carved(size_t b) { return (b + 255) & ~size_t(255); }

// Buffers of a sample sort, carved from one scratch.
struct SplitBufs {
    unsigned long long *pa, *pb, *kcopy;
    SplitTable *tab1, *tab2;
    unsigned *ia, *ib, *size1, *size2, *wide_n, *start1, *cur1, *start2, *cur2;
    unsigned short* ids;
    uint4 *rec, *wide;
    size_t zeroed, bytes;  // the counters lie together: bytes to clear from size1 on
    unsigned wide_cap;
};
static SplitBufs carve_split(void* scratch, unsigned W, unsigned long long n, unsigned long long windows,
                             const SplitPlan& pl) {
    unsigned char* const p0 = static_cast<unsigned char*>(scratch);
    size_t off = 0;
    auto carve = [&](size_t bytes) {
        unsigned char* r = p0 + off;
        off += carved(bytes);
        return r;
    };
    SplitBufs b{};
    const size_t f1 = pl.fan1, f12 = (size_t)pl.fan1 * pl.fan2;
    b.wide_cap = (unsigned)(windows / 65536 + 1);
    b.rec = reinterpret_cast<uint4*>(carve(n * 16 * kSlimU4));
    b.wide = reinterpret_cast<uint4*>(carve((size_t)b.wide_cap * 32));
    if (W >= 2) b.kcopy = reinterpret_cast<unsigned long long*>(carve(n * 8 * W));
    const size_t z0 = off;
    b.size1 = reinterpret_cast<unsigned*>(carve((f1 + 1) * 4));
    b.size2 = reinterpret_cast<unsigned*>(carve(f12 * 4));
    b.wide_n = reinterpret_cast<unsigned*>(carve(4));
    b.zeroed = off - z0;
    if (pl.levels >= 1) {
        b.ids = reinterpret_cast<unsigned short*>(carve(n * 2));
        b.pa = reinterpret_cast<unsigned long long*>(carve(n * 8));
        b.ia = reinterpret_cast<unsigned*>(carve(n * 4));
        b.tab1 = reinterpret_cast<SplitTable*>(carve(sizeof(SplitTable)));
        b.start1 = reinterpret_cast<unsigned*>(carve((f1 + 1) * 4));
        b.cur1 = reinterpret_cast<unsigned*>(carve(f1 * 4));
    }
    if (pl.levels >= 2 || (pl.levels >= 1 && W >= 2)) b.pb = reinterpret_cast<unsigned long long*>(carve(n * 8));
    if (pl.levels >= 2) {
        b.ib = reinterpret_cast<unsigned*>(carve(n * 4));
        b.tab2 = reinterpret_cast<SplitTable*>(carve(f1 * sizeof(SplitTable)));
        b.start2 = reinterpret_cast<unsigned*>(carve((f12 + 1) * 4));
        b.cur2 = reinterpret_cast<unsigned*>(carve(f12 * 4));
    }
    b.bytes = off;
    return b;
}

template <int W>
static cudaError_t sample_sort_w(unsigned long long* keys, unsigned* count, unsigned* ext, unsigned char* cls,
                                 unsigned long long n64, unsigned long long windows, unsigned k, void* scratch,
                                 unsigned* status, int num_sms, unsigned* launches, cudaStream_t s) {
    const SplitPlan pl = split_plan(n64, num_sms);
    const SplitBufs b = carve_split(scratch, W, n64, windows, pl);
    const unsigned n = (unsigned)n64, hb = 2 * k - 64 * (W - 1);
    constexpr size_t kScatterSmem = kSplitTile * 14, kBucketSmem = kBucketCap * 12 + (kLut + 4) * 4;
    cudaError_t e = cudaMemsetAsync(b.size1, 0, b.zeroed, s);
    if (e != cudaSuccess) return e;
    auto pick_smem = [](unsigned fan, unsigned over) { return (size_t)fan * over * 8; };
    if (pl.levels) {
        const size_t ps = pick_smem(pl.fan1, pl.over1);
        e = raise_smem_limit((const void*)split_pick_kernel<W>, ps);
        if (e != cudaSuccess) return e;
        split_pick_kernel<W><<<1, kPickThreads, ps, s>>>(keys, nullptr, n, hb, (n + pl.fan1 - 1) / pl.fan1, pl.over1,
                                                         pl.fan1, b.tab1);
        ++*launches;
    }
    const unsigned long long cb = (n64 + kSplitThreads - 1) / kSplitThreads;
    const unsigned cgrid = (unsigned)(cb < (unsigned long long)num_sms * 8 ? cb : num_sms * 8);
    sort_count1_kernel<W><<<cgrid, kSplitThreads, 0, s>>>(keys, count, ext, cls, n, hb, b.tab1, pl.levels ? pl.fan1 : 1u,
                                                         b.ids, pl.levels ? b.pb : nullptr, b.kcopy, b.rec, b.wide,
                                                         b.wide_n, b.wide_cap, b.size1, status);
    ++*launches;
    const unsigned long long* src = nullptr;
    const unsigned *pos = nullptr, *bstart = nullptr;
    unsigned buckets = 1;
    if (pl.levels) {
        e = raise_smem_limit((const void*)sort_scatter_kernel<0>, kScatterSmem);
        if constexpr (W == 1)
            if (e == cudaSuccess) e = raise_smem_limit((const void*)sort_scatter_kernel<1>, kScatterSmem);
        if (e != cudaSuccess) return e;
        sort_starts_kernel<<<1, kSplitThreads, 0, s>>>(b.size1, nullptr, n, pl.fan1,
                                                       pl.levels == 1 ? kBucketCap : 0xFFFFFFFFu, b.start1, b.cur1, status);
        const unsigned long long tiles = (n64 + kSplitTile - 1) / kSplitTile + pl.fan1;
        const unsigned sgrid = (unsigned)(tiles < (unsigned long long)num_sms * 3 ? tiles : num_sms * 3);
        if constexpr (W == 1)
            sort_scatter_kernel<1><<<sgrid, kSplitThreads, kScatterSmem, s>>>(keys, nullptr, b.ids, nullptr, 1, n, hb,
                                                                             pl.fan1, b.cur1, b.pa, b.ia);
        else
            sort_scatter_kernel<0><<<sgrid, kSplitThreads, kScatterSmem, s>>>(b.pb, nullptr, b.ids, nullptr, 1, n, hb,
                                                                             pl.fan1, b.cur1, b.pa, b.ia);
        *launches += 2;
        src = b.pa;
        pos = b.ia;
        bstart = b.start1;
        buckets = pl.fan1;
        if (pl.levels == 2) {
            const unsigned over = kMaxSamples / pl.fan2 < 32 ? kMaxSamples / pl.fan2 : 32;
            const size_t ps = pick_smem(pl.fan2, over);
            e = raise_smem_limit((const void*)split_pick_kernel<0>, ps);
            if (e != cudaSuccess) return e;
            split_pick_kernel<0><<<pl.fan1, kPickThreads, ps, s>>>(b.pa, b.start1, n, hb, pl.mean, over, pl.fan2, b.tab2);
            sort_count2_kernel<<<num_sms * 4, kSplitThreads, 0, s>>>(b.pa, b.start1, pl.fan1, b.tab2, pl.mean, pl.fan2,
                                                                     b.ids, b.size2);
            sort_starts_kernel<<<pl.fan1, kSplitThreads, 0, s>>>(b.size2, b.start1, n, pl.fan2, kBucketCap, b.start2,
                                                                 b.cur2, status);
            sort_scatter_kernel<0><<<sgrid, kSplitThreads, kScatterSmem, s>>>(b.pa, b.ia, b.ids, b.start1, pl.fan1, n, hb,
                                                                             pl.fan2, b.cur2, b.pb, b.ib);
            *launches += 4;
            src = b.pb;
            pos = b.ib;
            bstart = b.start2;
            buckets = pl.fan1 * pl.fan2;
        }
    }
    e = raise_smem_limit((const void*)sort_buckets_kernel<W>, kBucketSmem);
    if (e != cudaSuccess) return e;
    sort_buckets_kernel<W><<<buckets, kSplitThreads, kBucketSmem, s>>>(src, pos, bstart, n, hb, b.kcopy, b.rec, b.wide,
                                                                      b.wide_cap, status, keys, count, ext, cls);
    ++*launches;
    return cudaGetLastError();
}

static unsigned sort_passes(unsigned k) { return (2 * k + 7) / 8; }

static unsigned long long sort_tiles(unsigned W, unsigned long long n) {
    const unsigned long long T = W == 1   ? SortShape<1>::TILE
                                 : W == 2 ? SortShape<2>::TILE
                                 : W == 3 ? SortShape<3>::TILE
                                          : SortShape<4>::TILE;
    return (n + T - 1) / T;
}

static size_t digit_scratch_bytes(unsigned W, unsigned long long n) {
    const unsigned passes = sort_passes(32 * W);  // enough for any k of this width
    return carved(n * 8 * W) + 2 * carved(n * 4) + carved(sort_tiles(W, n) * 256 * 8) + carved(passes * 256 * 4) +
           carved(passes * 4) + carved(n * 16 * kRecU4);
}

size_t sort_scratch_bytes(unsigned W, unsigned long long n, unsigned long long windows, int num_sms) {
    const size_t d = digit_scratch_bytes(W, n);
    if (n > kSampleSortMax) return d;
    return std::max(d, carve_split(nullptr, W, n, windows, split_plan(n, num_sms)).bytes);
}

template <int W>
static cudaError_t sort_w(unsigned long long* keys, unsigned* count, unsigned* ext, unsigned char* cls,
                          unsigned long long n, unsigned k, void* scratch, unsigned* status, int num_sms,
                          unsigned* launches, cudaStream_t s) {
    using Shape = SortShape<W>;
    const unsigned long long tiles = (n + Shape::TILE - 1) / Shape::TILE;
    const unsigned passes = sort_passes(k);
    unsigned char* p = static_cast<unsigned char*>(scratch);
    auto carve = [&](size_t bytes) {
        unsigned char* r = p;
        p += carved(bytes);
        return r;
    };
    unsigned long long* kb = reinterpret_cast<unsigned long long*>(carve(n * 8 * W));
    unsigned* ia = reinterpret_cast<unsigned*>(carve(n * 4));
    unsigned* ib = reinterpret_cast<unsigned*>(carve(n * 4));
    unsigned long long* st = reinterpret_cast<unsigned long long*>(carve(tiles * 256 * 8));
    unsigned* hist = reinterpret_cast<unsigned*>(carve(passes * 256 * 4));
    unsigned* counters = reinterpret_cast<unsigned*>(carve(passes * 4));
    uint4* rec = reinterpret_cast<uint4*>(carve(n * 16 * kRecU4));
    cudaError_t e = cudaMemsetAsync(st, 0, tiles * 256 * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(hist, 0, passes * 256 * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(counters, 0, passes * 4, s);
    if (e != cudaSuccess) return e;
    // digit totals of every pass (passes whose digit is the same for every key
    // move nothing) and the payload records
    const size_t hsmem = passes * 256 * 4;
    e = raise_smem_limit((const void*)sort_digits_kernel<W>, hsmem);
    if (e != cudaSuccess) return e;
    const unsigned long long hb = (n + kSortThreads - 1) / kSortThreads;
    const unsigned hgrid = (unsigned)(hb < (unsigned long long)num_sms * 16 ? hb : num_sms * 16);
    sort_digits_kernel<W><<<hgrid, kSortThreads, hsmem, s>>>(keys, count, ext, cls, n, passes, hist, rec);
    ++*launches;
    std::vector<unsigned> h(passes * 256);
    e = cudaMemcpyAsync(h.data(), hist, h.size() * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    e = raise_smem_limit((const void*)sort_pass_kernel<W>, Shape::SMEM);
    if (e != cudaSuccess) return e;
    // keys move from `keys` to the scratch and back, pass by pass (a final
    // copy into `keys` when the number of passes that moved is odd)
    const unsigned long long* src = keys;
    const unsigned* isrc = nullptr;
    unsigned long long* bufs[2] = {kb, keys};
    unsigned* ibufs[2] = {ia, ib};
    unsigned moved = 0;
    for (unsigned pass = 0; pass < passes; ++pass) {
        unsigned nz = 0;
        for (int d = 0; d < 256; ++d) nz += h[pass * 256 + d] != 0;
        if (nz <= 1) continue;
        unsigned long long* dst = bufs[moved & 1];
        unsigned* idst = ibufs[moved & 1];
        sort_pass_kernel<W><<<(unsigned)tiles, kSortThreads, Shape::SMEM, s>>>(
            src, isrc, n, pass, moved, hist, st, counters + pass, dst, idst, status);
        ++*launches;
        src = dst;
        isrc = idst;
        ++moved;
    }
    if (!moved) return cudaGetLastError();  // a single key value: nothing moves
    if (src != keys) {
        e = cudaMemcpyAsync(keys, src, n * 8 * W, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return e;
    }
    const unsigned long long gb = (n + 255) / 256;
    const unsigned g = (unsigned)(gb < (unsigned long long)num_sms * 32 ? gb : num_sms * 32);
    sort_gather_kernel<<<g, 256, 0, s>>>(isrc, n, rec, count, ext, cls);
    ++*launches;
    return cudaGetLastError();
}

static bool sortable(unsigned W, const unsigned long long* keys, const unsigned* count, const unsigned* ext,
                     const unsigned char* cls, unsigned long long n, unsigned k) {
    return n < 0xFFFFFFFFull && (2 * k + 63) / 64 == W && !(reinterpret_cast<uintptr_t>(keys) & 7) &&
           !(reinterpret_cast<uintptr_t>(count) & 3) && !(reinterpret_cast<uintptr_t>(ext) & 15) &&
           !(reinterpret_cast<uintptr_t>(cls) & 1);
}

cudaError_t launch_sort_by_digits(unsigned W, unsigned long long* keys, unsigned* count, unsigned* ext,
                                  unsigned char* cls, unsigned long long n, unsigned k, void* scratch,
                                  unsigned* status, int num_sms, unsigned* launches, cudaStream_t s) {
    if (n < 2) return cudaSuccess;
    if (!sortable(W, keys, count, ext, cls, n, k)) return cudaErrorInvalidValue;
    switch (W) {
        case 1: return sort_w<1>(keys, count, ext, cls, n, k, scratch, status, num_sms, launches, s);
        case 2: return sort_w<2>(keys, count, ext, cls, n, k, scratch, status, num_sms, launches, s);
        case 3: return sort_w<3>(keys, count, ext, cls, n, k, scratch, status, num_sms, launches, s);
        case 4: return sort_w<4>(keys, count, ext, cls, n, k, scratch, status, num_sms, launches, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_sort_survivors(unsigned W, unsigned long long* keys, unsigned* count, unsigned* ext,
                                  unsigned char* cls, unsigned long long n, unsigned long long windows, unsigned k,
                                  void* scratch, unsigned* status, int num_sms, unsigned* launches, cudaStream_t s) {
    if (n < 2) return cudaSuccess;
    if (!sortable(W, keys, count, ext, cls, n, k)) return cudaErrorInvalidValue;
    if (n > kSampleSortMax)
        return launch_sort_by_digits(W, keys, count, ext, cls, n, k, scratch, status, num_sms, launches, s);
    switch (W) {
        case 1: return sample_sort_w<1>(keys, count, ext, cls, n, windows, k, scratch, status, num_sms, launches, s);
        case 2: return sample_sort_w<2>(keys, count, ext, cls, n, windows, k, scratch, status, num_sms, launches, s);
        case 3: return sample_sort_w<3>(keys, count, ext, cls, n, windows, k, scratch, status, num_sms, launches, s);
        case 4: return sample_sort_w<4>(keys, count, ext, cls, n, windows, k, scratch, status, num_sms, launches, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kmer
