// Level-1 scatter: one thread per read rolls its k-windows (a2, a3), turns
// each into a W-word record and hands it to the level-1 bucket picked by the
// top bits of the mixed key.  This is the all-to-all k-mer exchange of the
// paper's k-mer analysis (Sec. II-B), done as a device-wide partition in HBM:
// a bucket plays the role of the owning processor.
//
// Bound by issue slots (integer work of the windows, then the staging of the
// records), not by DRAM.  A thread starts at its read's first window (Roll)
// and a round's steps are unrolled, so the records' meta words stay in
// registers; three CTAs per SM.  2-Gbase reads at k = 31: 11.45 -> 9.08 ms
// (176 G windows/s); 300 Mbases at k = 99: 3.05 -> 1.21 ms; 100 Mbases at
// k = 77: 1.43 -> 0.92 ms.  512 threads and 8 positions a round: 10.4 ms.
#include "kernels.h"
#include "roll.cuh"
#include "stage.cuh"

namespace kmer {

template <int W>
struct ScatterShape {
    // threads of a CTA (three CTAs per SM), read positions per round, staged records per round
    static constexpr unsigned NT = 256, CTAS = 3;
    static constexpr unsigned R = W == 1 ? 16 : (W == 2 ? 10 : (W == 3 ? 8 : 7));
    static_assert(NT == 256, "one tile size for every width");
    static constexpr unsigned S = R * NT;
};

struct L1Dest {
    unsigned long long* fill;
    const unsigned long long* startp;
    const unsigned long long* capp;
    __device__ unsigned long long reserve(unsigned d, unsigned n) { return atomicAdd(fill + d, (unsigned long long)n); }
    __device__ unsigned long long start(unsigned d) const { return __ldg(startp + d); }
    __device__ unsigned long long cap(unsigned d) const { return __ldg(capp + d); }
};

// One CTA: the reads [r0, r1) of job j (a read tile), NT >> seg_bits of them at
// most: 2^seg_bits threads share a read, each taking a run of its windows (the
// threads of a warp take the same run of their reads).
// MAXPER: destinations handled by one thread in a flush (fan-out / NT).
template <int W, unsigned MAXPER, bool HI, bool GATE>
__device__ __forceinline__ void scatter_tile(const Job& j, const unsigned long long r0, const unsigned long long r1,
                                             const unsigned seg_bits, unsigned char* smem) {
    constexpr unsigned R = ScatterShape<W>::R, S = ScatterShape<W>::S, NT = ScatterShape<W>::NT;
    __shared__ unsigned s_steps;
    const unsigned P = 1u << j.g.p1;
    StageBufs b = carve_stage(smem, W, S, P);
    if (threadIdx.x == 0) s_steps = 0;
    for (unsigned d = threadIdx.x; d < P; d += NT) b.hist[d] = 0;
    __syncthreads();

    const unsigned tile = NT >> seg_bits;
    const unsigned long long r = r0 + threadIdx.x % tile;
    const Geometry g = j.g;
    Roll<W, HI> roll;
    unsigned t = 0, end = 0;  // this thread's steps [t, end)
    if (r < r1) {
        const unsigned long long L = j.offsets[r + 1] - j.offsets[r];  // below 2^31
        if (L >= g.k) {
            const unsigned n = (unsigned)L - g.k + 1, per = (n + (1u << seg_bits) - 1) >> seg_bits;
            const unsigned w0 = per * (threadIdx.x / tile);
            if (w0 < n) {
                roll.init(j, r, w0);
                t = g.k + w0;
                end = t + (per < n - w0 ? per : n - w0);
                atomicMax(&s_steps, end - t);
            }
        }
    }
    __syncthreads();
    const unsigned steps = s_steps;
    L1Dest dest{j.l1_fill, j.l1_start, j.l1_cap};
    const unsigned pass = j.pass;
    const unsigned long long* gate = j.gate;  // Bloom gate (GATE): emit only keys in F2
    const unsigned long long gate_words = j.gate_words;
    unsigned emitted = 0;
    for (unsigned s0 = 0; s0 < steps; s0 += R) {
        unsigned m[R];
#pragma unroll
        for (unsigned s = 0; s < R; ++s) {
            const unsigned e = s * NT + threadIdx.x;
            m[s] = 0xFFFFFFFFu;
            if (t < end) {
                unsigned long long key[W], rec[W];
                unsigned lc = 0, rc = 0, bucket = 0;
                if (roll.step(t++, key, lc, rc) && (!GATE || gate_has<W>(gate, gate_words, key)) &&
                    make_record<W>(g, pass, key, lc, rc, rec, bucket)) {
                    m[s] = (bucket << 16) | atomicAdd(&b.hist[bucket], 1u);
                    if constexpr (W == 2 || W == 4) {
#pragma unroll
                        for (int w = 0; w < W; w += 2)
                            *reinterpret_cast<ulonglong2*>(b.stage + (size_t)e * W + w) = make_ulonglong2(rec[w], rec[w + 1]);
                    } else {
#pragma unroll
                        for (int w = 0; w < W; ++w) b.stage[(size_t)e * W + w] = rec[w];
                    }
                    ++emitted;
                }
            }
        }
        flush_stage_regs<W, MAXPER, L1Dest, NT, R>(b, S, P, dest, j.l1_rec, j.status, ST_L1_OVERFLOW, m);
    }
    // windows emitted into this pass (checked against the windows the leaves count)
#pragma unroll
    for (int o = 16; o; o >>= 1) emitted += __shfl_xor_sync(0xffffffffu, emitted, o);
    if ((threadIdx.x & 31) == 0 && emitted) atomicAdd(j.stats + 2, (unsigned long long)emitted);
}

// One CTA per read tile over all jobs (all of key width W).
template <int W, unsigned MAXPER, bool HI, bool GATE>
__global__ void __launch_bounds__(ScatterShape<W>::NT, ScatterShape<W>::CTAS)
scatter_kernel(const Job* __restrict__ jobs, const unsigned long long* __restrict__ tile_off, const unsigned n_jobs,
               const unsigned seg_bits) {
    const unsigned tile = ScatterShape<W>::NT >> seg_bits;
    extern __shared__ __align__(16) unsigned char smem[];
    const unsigned long long t = blockIdx.x;
    const unsigned ji = job_of(tile_off, n_jobs, t);
    const Job& j = jobs[ji];
    const unsigned long long r0 = (t - tile_off[ji]) * tile;
    const unsigned long long r1 = r0 + tile < j.n_reads ? r0 + tile : j.n_reads;
    scatter_tile<W, MAXPER, HI, GATE>(j, r0, r1, seg_bits, smem);
}

// Threads that share a read, as a power of two: as many (up to eight) as it
// takes to give every SM its three CTAs.  20 000 reads are 79 tiles of one
// thread per read, half of the SMs idle and each tile ten rounds long (65-100
// us at k = 21 to 99; 29-39 us with eight threads a read).
unsigned scatter_seg_bits(unsigned long long n_reads, int num_sms) {
    unsigned b = 0;
    while (b < 3 && (n_reads << b) < 3ull * num_sms * ScatterShape<1>::NT) ++b;
    return b;
}
unsigned scatter_tile_reads(unsigned seg_bits) { return ScatterShape<1>::NT >> seg_bits; }

size_t scatter_smem_bytes(unsigned W, unsigned p1) {
    const unsigned P = 1u << p1;
    switch (W) {
        case 1: return stage_smem_bytes(1, ScatterShape<1>::S, P);
        case 2: return stage_smem_bytes(2, ScatterShape<2>::S, P);
        case 3: return stage_smem_bytes(3, ScatterShape<3>::S, P);
        default: return stage_smem_bytes(4, ScatterShape<4>::S, P);
    }
}

template <int W, unsigned MAXPER, bool HI, bool GATE>
static cudaError_t launch_scatter_wpg(const Job* jobs, const unsigned long long* tile_off, unsigned n_jobs,
                                      unsigned long long tiles, unsigned seg_bits, unsigned max_p1, cudaStream_t s) {
    const size_t smem = scatter_smem_bytes(W, max_p1);
    cudaError_t e = raise_smem_limit((const void*)scatter_kernel<W, MAXPER, HI, GATE>, smem);
    if (e != cudaSuccess) return e;
    if (tiles == 0) return cudaSuccess;
    if (tiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    scatter_kernel<W, MAXPER, HI, GATE><<<(unsigned)tiles, ScatterShape<W>::NT, smem, s>>>(jobs, tile_off, n_jobs, seg_bits);
    return cudaGetLastError();
}

template <int W, unsigned MAXPER, bool HI>
static cudaError_t launch_scatter_wp(const Job* jobs, const unsigned long long* tile_off, unsigned n_jobs,
                                     unsigned long long tiles, unsigned seg_bits, unsigned max_p1, bool gated,
                                     cudaStream_t s) {
    return gated ? launch_scatter_wpg<W, MAXPER, HI, true>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, s)
                 : launch_scatter_wpg<W, MAXPER, HI, false>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, s);
}

template <int W, bool HI>
static cudaError_t launch_scatter_w(const Job* jobs, const unsigned long long* tile_off, unsigned n_jobs,
                                    unsigned long long tiles, unsigned seg_bits, unsigned max_p1, bool gated,
                                     cudaStream_t s) {
    // MAXPER: destinations of one thread in a flush (fan-out / threads, rounded up)
    constexpr unsigned NT = ScatterShape<W>::NT;
    if ((1u << max_p1) <= 2 * NT)
        return launch_scatter_wp<W, 2, HI>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
    if constexpr (kMaxStageDest / NT > 4)
        if ((1u << max_p1) <= 4 * NT)
            return launch_scatter_wp<W, 4, HI>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
    return launch_scatter_wp<W, kMaxStageDest / NT, HI>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
}

cudaError_t launch_scatter(unsigned W, const Job* jobs, const unsigned long long* tile_off, unsigned n_jobs,
                           unsigned long long tiles, unsigned seg_bits, unsigned max_p1, unsigned min_k, bool gated,
                           cudaStream_t s) {
    switch (W) {
        case 1:
            return min_k >= 17 ? launch_scatter_w<1, true>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s)
                               : launch_scatter_w<1, false>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
        case 2: return launch_scatter_w<2, false>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
        case 3: return launch_scatter_w<3, false>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
        case 4: return launch_scatter_w<4, false>(jobs, tile_off, n_jobs, tiles, seg_bits, max_p1, gated, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kmer
