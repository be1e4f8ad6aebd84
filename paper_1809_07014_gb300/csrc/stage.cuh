// Shared-memory staging of partitioned records: records of one round are
// counted per destination in shared memory, one global atomic per
// destination reserves their slots, and the records are written out sorted
// by destination so that each warp stores contiguous runs.  This is the
// aggregation of fine-grained inserts into batch updates that the paper
// describes for update-only hash-table phases (Sec. II-A, use case 1).
#pragma once
#include "common.cuh"

namespace kmer {

constexpr int kStageThreads = 256;
constexpr unsigned kMaxStageDest = 2048;  // destinations of one staging round (partition fan-out)

// Exclusive scan across the kStageThreads threads of the block (all must call; warp_tmp holds 8 words).
__device__ inline unsigned long long block_scan_u64(unsigned long long v, unsigned long long* warp_tmp,
                                                    unsigned long long* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tmp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long s = lane < kStageThreads / 32 ? warp_tmp[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kStageThreads / 32) warp_tmp[lane] = s;
    }
    __syncthreads();
    const unsigned long long before = wid ? warp_tmp[wid - 1] : 0ull;
    *total = warp_tmp[kStageThreads / 32 - 1];
    __syncthreads();
    return before + x - v;
}

struct StageBufs {
    unsigned long long* stage;   // S * W: records in arrival order
    unsigned long long* wbase;   // P: record index of sorted position 0 of destination d
    unsigned* ok_end;            // P: first sorted position of destination d past its capacity
    unsigned* hist;              // P
    unsigned* lbase;             // P
    unsigned* order;             // S: (destination << 16) | staged index, per sorted position
    unsigned* warp_tmp;          // one word per warp of the block (up to 32)
};

__host__ __device__ inline size_t stage_smem_bytes(unsigned W, unsigned S, unsigned P) {
    return (size_t)S * W * 8 + (size_t)P * 8 + (size_t)P * 4 + (size_t)P * 8 + (size_t)S * 4 + 128;
}

__device__ inline StageBufs carve_stage(unsigned char* base, unsigned W, unsigned S, unsigned P) {
    StageBufs b;
    b.stage = reinterpret_cast<unsigned long long*>(base);
    b.wbase = b.stage + (size_t)S * W;
    b.ok_end = reinterpret_cast<unsigned*>(b.wbase + P);
    b.hist = b.ok_end + P;
    b.lbase = b.hist + P;
    b.order = b.lbase + P;
    b.warp_tmp = b.order + S;
    return b;
}

// Flush one round.  A staged record e has the meta word (dest << 16) | rank, or
// 0xFFFFFFFF for none; hist[d] = records staged for destination d (S <= 65536).  Dest
// supplies reserve(d, n) -> first slot index within d, start(d) -> record
// index of slot 0 of d, cap(d) -> slots of d.  Records past cap are dropped
// and reported through `status` (the host then retries with exact
// capacities).  hist is left zeroed for the next round.
//
// The records are not moved inside shared memory: a word per sorted position
// says which staged record goes there and to which destination, and
// consecutive threads write consecutive positions, i.e. contiguous runs per
// destination.
//
// Five barriers a flush, each destination's count read (and cleared) once;
// whether any record lacks room is known to the whole block before the
// writes, so the usual flush does not look at the destinations' limits.
//
// `sort` places every staged record's word in `order` once the local bases
// are known (from the meta words the threads keep in registers).
template <int W, unsigned MAXPER, class Dest, unsigned NT, class Sort>
__device__ __forceinline__ void flush_stage_with(const StageBufs& b, unsigned S, unsigned P, Dest& dest,
                                                 unsigned long long* out_rec, unsigned* status,
                                                 unsigned overflow_bit, Sort sort) {
    __syncthreads();
    // exclusive scan of hist -> lbase (each thread owns a run of consecutive
    // destinations, at most MAXPER); hist is cleared as it is read
    const unsigned per = (P + NT - 1) / NT;
    const unsigned d0 = threadIdx.x * per;
    unsigned hs[MAXPER], mine = 0;
#pragma unroll
    for (unsigned i = 0; i < MAXPER; ++i) {
        hs[i] = 0;
        if (i < per && d0 + i < P) {
            hs[i] = b.hist[d0 + i];
            b.hist[d0 + i] = 0;
        }
        mine += hs[i];
    }
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (unsigned)o) x += y;
    }
    if (lane == 31) b.warp_tmp[wid] = x;
    __syncthreads();
    // every warp scans the warps' totals itself
    unsigned wt = lane < NT / 32 ? b.warp_tmp[lane] : 0u;
#pragma unroll
    for (unsigned o = 1; o < NT / 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, wt, o);
        if (lane >= o) wt += y;
    }
    const unsigned total = __shfl_sync(0xffffffffu, wt, NT / 32 - 1);
    const unsigned before = __shfl_sync(0xffffffffu, wt, wid ? wid - 1 : 0);
    const unsigned run0 = (wid ? before : 0u) + x - mine;
    // reservations of this thread's destinations are independent: all are
    // issued together, and their results are only used after the sort below
    // (which needs just the local bases), so the atomics' latency overlaps it
    unsigned long long first[MAXPER];
    unsigned run = run0;
#pragma unroll
    for (unsigned i = 0; i < MAXPER; ++i) {
        first[i] = 0;
        if (i < per && d0 + i < P) {
            b.lbase[d0 + i] = run;
            if (hs[i]) first[i] = dest.reserve(d0 + i, hs[i]);
            run += hs[i];
        }
    }
    __syncthreads();
    sort();
    bool over = false;
    run = run0;
#pragma unroll
    for (unsigned i = 0; i < MAXPER; ++i) {
        const unsigned d = d0 + i;
        const unsigned h = hs[i];
        if (h) {
            const unsigned long long cap = dest.cap(d);
            b.wbase[d] = dest.start(d) + first[i] - run;
            // positions of d that still fit: [run, run + min(h, cap - first))
            const unsigned long long room = first[i] < cap ? cap - first[i] : 0ull;
            b.ok_end[d] = run + (unsigned)(room < h ? room : h);
            over = over || room < h;
        }
        run += h;
    }
    const bool check = __syncthreads_or(over);  // some record of the round has no room
    // two-word records move as 16-byte words, four-word ones as two of them by
    // neighbouring threads, three-word ones word by word: a warp's stores stay
    // consecutive
    constexpr unsigned PARTS = W <= 2 ? 1 : (W == 4 ? 2 : 3);
    for (unsigned i = threadIdx.x; i < total * PARTS; i += NT) {
        const unsigned pos = i / PARTS, part = i % PARTS;
        const unsigned o = b.order[pos];
        const unsigned d = o >> 16, e = o & 0xFFFFu;
        if (!check || pos < b.ok_end[d]) {
            const unsigned long long g = b.wbase[d] + pos;
            if constexpr (W == 1 || W == 3)
                out_rec[g * PARTS + part] = b.stage[(size_t)e * PARTS + part];
            else
                reinterpret_cast<ulonglong2*>(out_rec)[g * PARTS + part] =
                    reinterpret_cast<const ulonglong2*>(b.stage)[(size_t)e * PARTS + part];
        }
    }
    if (over) atomicOr(status, overflow_bit);
    __syncthreads();
}

// Sorted position of staged record e with meta word m (see flush_stage).
__device__ __forceinline__ void place(const StageBufs& b, unsigned m, unsigned e) {
    if (m != 0xFFFFFFFFu) b.order[b.lbase[m >> 16] + (m & 0xFFFFu)] = (m & 0xFFFF0000u) | e;
}

// Meta words in registers: m[u] belongs to staged record u * NT + threadIdx.x.
template <int W, unsigned MAXPER, class Dest, unsigned NT, unsigned U>
__device__ void flush_stage_regs(const StageBufs& b, unsigned S, unsigned P, Dest& dest, unsigned long long* out_rec,
                                 unsigned* status, unsigned overflow_bit, const unsigned (&m)[U]) {
    flush_stage_with<W, MAXPER, Dest, NT>(b, S, P, dest, out_rec, status, overflow_bit, [&]() {
#pragma unroll
        for (unsigned u = 0; u < U; ++u) place(b, m[u], u * NT + threadIdx.x);
    });
}

}  // namespace kmer
