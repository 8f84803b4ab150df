// Bands of levels: what the clique peel and the star peel share.
//
// A band is the run of consecutive levels that one cascade (remove everything
// below a threshold, repeat) takes out of the alive set.
#pragma once

#include "common.cuh"

namespace dsd {

constexpr uint32_t kMaxBands = 4096;    // multi-level bands (then levels go one by one)
// A threshold is set for at most kBandAim vertices, or fewer (pick_threshold);
// a cascade that removes more than kBandMax is undone and its first level
// taken alone: a band's owner block reads all its members every round.
constexpr uint32_t kBandAim = 2048;
constexpr uint32_t kBandMax = 8192;
// A cascade longer than kBandRounds is undone likewise: it runs along a path
// of the graph, one level's worth of rounds or nearly, and phase 2 would run
// them all again (a strip of 3,000 triangles, h = 3, 1,500 rounds in one level:
// the call 26.6 ms, 20.1 undone after 48).  On the power-law, R-MAT and
// Erdos-Renyi graphs measured, h = 2..5, no cascade takes more than 30.
constexpr uint32_t kBandRounds = 48;
// With N vertices left a band aims at sqrt(kBandFill N) of them: a cascade
// takes 2-5 rounds, so phase 1 runs ~3 N / T rounds for bands of T vertices and
// phase 2 as many as the fullest band has levels (up to one a vertex).  The
// 1M-vertex graph (h = 3) and R-MAT scale 17 (h = 4) take the same time within
// 3 % from 1 to 16.
constexpr float kBandFill = 2.0f;
// ... and never at more than kBandAim: from 33.5M vertices on a first frontier
// alone could pass kBandMax, so that every cascade would be undone.
__device__ __forceinline__ uint32_t band_aim(uint32_t left) {
    const uint32_t t = (uint32_t)sqrtf(kBandFill * (float)left);
    return t < kBandAim ? t : kBandAim;
}

// Warp-aggregated append of `val` where pred holds (all lanes call).
__device__ __forceinline__ void warp_append(bool pred, uint32_t val, uint32_t* counter,
                                            uint32_t* list) {
    unsigned lane = lane_id();
    unsigned b = __ballot_sync(0xffffffffu, pred);
    if (!b) return;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(counter, (uint32_t)__popc(b));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (pred) list[base + __popc(b & ((1u << lane) - 1u))] = val;
}

// Block-wide exclusive scan of small per-thread counts; returns this
// thread's prefix and the total in *tot (all threads).
template <int NT>
__device__ __forceinline__ uint32_t block_scan_count(uint32_t v, uint32_t* wtot, uint32_t* tot) {
    unsigned lane = lane_id(), wid = warp_id();
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane >= o) x += y;
    }
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int w = 0; w < NT / 32; w++) {
        uint32_t t = wtot[w];
        before += (w < (int)wid) ? t : 0u;
        all += t;
    }
    __syncthreads();
    *tot = all;
    return before + x - v;
}

// Histogram of count offsets at a jump: 16 bins an octave, exact below 32.
constexpr uint32_t kBins = 1024;
constexpr uint32_t kLastBin = 975;      // the bin of 2^64 - 1
__device__ __forceinline__ uint32_t bin_of(unsigned long long d) {
    if (d < 16) return (uint32_t)d;
    const uint32_t e = 63u - (uint32_t)__clzll((long long)d);
    return (e - 3u) * 16u + ((uint32_t)(d >> (e - 4u)) & 15u);
}
// Largest offset of bin b <= kLastBin.
__device__ __forceinline__ unsigned long long bin_last(uint32_t b) {
    if (b < 16) return b;
    const uint32_t e = (b >> 4) + 3u;
    return (((16ull + (b & 15u)) + 1ull) << (e - 4u)) - 1ull;
}

// A multi-level band: members mem[seg .. seg + size).
struct Band {
    unsigned long long k;           // phase 2: current level
    unsigned long long mu;          // cliques of the current set (the band and above)
    uint32_t seg, size;
    uint32_t left;                  // size; 0 once every member has left
    uint32_t above;                 // vertices of the bands above
    uint32_t nlev, rounds;
    uint32_t rbase;                 // single-level rounds of phase 1 before the band
    uint32_t pad;
};

// The threshold of a jump (every block alike): the largest count k + 1 + hi
// such that the alive vertices at or below it number at most `tmax`, or at
// most kBandAim and span at most `lmax` values.  hist: the alive vertices by bin_of(count - k - 1).
// Returns k + 1 + hi, or 0 when even the first occupied bin is larger.
template <int NT>
__device__ __forceinline__ unsigned long long pick_threshold(const uint32_t* hist,
                                                             unsigned long long k, uint32_t tmax,
                                                             uint32_t lmax, uint32_t* s_wtot,
                                                             uint32_t* s_best) {
    constexpr uint32_t E = kBins / NT > 0 ? kBins / NT : 1;
    static_assert(kBins % NT == 0, "a whole number of bins per thread");
    uint32_t c[E], sum = 0;
#pragma unroll
    for (uint32_t q = 0; q < E; q++) {
        c[q] = hist[threadIdx.x * E + q];
        sum += c[q];
    }
    if (threadIdx.x == 0) *s_best = 0;
    uint32_t tot;
    uint32_t run = block_scan_count<NT>(sum, s_wtot, &tot);
#pragma unroll
    for (uint32_t q = 0; q < E; q++) {
        const uint32_t b = threadIdx.x * E + q;
        run += c[q];
        // at least one vertex up to here, and few enough of them or of levels
        if (run && c[q] && (run <= tmax ||
                            (run <= kBandAim && bin_last(b < kLastBin ? b : kLastBin) < lmax)))
            atomicMax(s_best, b + 1);
    }
    __syncthreads();
    const uint32_t b = *s_best;
    __syncthreads();
    if (b == 0) return 0;
    const unsigned long long last = bin_last(b - 1);
    return last > ~0ull - k - 1 ? ~0ull : k + 1 + last;
}

}  // namespace dsd
