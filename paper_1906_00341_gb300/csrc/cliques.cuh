// Device routines shared by clique listing and peeling.
//
// Both reduce to one sub-problem: a fixed clique prefix ("root") and a
// sorted candidate list C of vertices adjacent to every root member; find
// the r-cliques inside G[C] and credit each member of C with the number of
// r-cliques it lies in (the root members get the total).  Each r-clique is
// listed once as an increasing sequence of positions in C, extending only
// through the oriented lists N+(x) = {y in N(x) : y > x}.  This is the
// kClist-style ordered listing the paper relies on for clique enumeration
// (Sec. 4.3), restated for warps and blocks.
//
// Local adjacency of G[C] is a bitmap: row i holds bit j (j > i) when C[j]
// is in N+(C[i]).  Up to 32 candidates a row is one word (warp routines);
// up to 1024 a row is 32 words, one per lane (block routines).
#pragma once

#include "common.cuh"

namespace dsd {

constexpr int kMaxDepth = DSD_MAX_H;     // r <= h - 1 <= 7
constexpr uint32_t kBitmapMax = 1024;   // candidates per bitmap problem

// ---------------------------------------------------------------------------
// Row construction: for candidate i, the positions j > i whose vertex is in
// N+(C[i]) = adj[nb[x] .. ne[x]).  Candidates are sorted ascending, N+ lists
// too, and every j > i automatically has C[j] > C[i]; membership is a binary
// search in C.

// Row scans read kScanChunks chunks of 32 entries per step (their loads in
// flight together) and stop at the first chunk past the largest candidate:
// the lists ascend, so nothing beyond it can be in C.
constexpr int kScanChunks = 4;

// Hits of the list adj[b, e) (ascending) in the sorted candidates C[0, nc)
// whose largest entry is cmax, by one warp: cnt[pos] += 1 for each hit
// (shared counters); returns this lane's number of hits.  Each step loads
// kScanChunks coalesced 32-entry chunks at once, lane l taking entry l of
// each, so that the lanes' binary searches look for neighbouring ids and
// follow nearly the same path through C; the scan stops after the first step
// that passes cmax.  *read_end (if given) receives the end of what was read.
template <class T>
__device__ __forceinline__ unsigned scan_row_hits(const uint32_t* C, uint32_t nc, uint32_t cmax,
                                                  const uint32_t* adj, uint64_t b, uint64_t e,
                                                  T* cnt, uint64_t* read_end = nullptr) {
    const unsigned lane = lane_id();
    unsigned hits = 0;
    uint64_t p0 = b;
    for (; p0 < e; p0 += 32 * kScanChunks) {
        uint32_t ys[kScanChunks];
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            ys[u] = p < e ? adj[p] : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            const uint32_t y = ys[u];
            if (y <= cmax) {
                uint32_t pos = (uint32_t)lower_bound_u32(C, nc, y);
                if (pos < nc && C[pos] == y) {
                    atomicAdd(&cnt[pos], (T)1);
                    hits++;
                }
            }
        }
        if (__shfl_sync(0xffffffffu, ys[kScanChunks - 1], 31) > cmax) {
            p0 += 32 * kScanChunks;
            break;
        }
    }
    if (read_end) *read_end = p0 < e ? p0 : e;
    return hits;
}

// One warp: the one-word row of candidate x = C[i] for |C| <= 32, i.e. bit j
// set iff C[j] > x lies in x's list adj[b, e) (sorted ascending; the scan
// stops past cmax = C[nc - 1]).  All lanes return it.
__device__ __forceinline__ uint32_t warp_row32(const uint32_t* C, uint32_t nc, uint32_t cmax,
                                               uint32_t x, const uint32_t* adj, uint64_t b,
                                               uint64_t e) {
    const unsigned lane = lane_id();
    uint32_t bits = 0;
    for (uint64_t p0 = b; p0 < e; p0 += 32 * kScanChunks) {
        uint32_t ys[kScanChunks];
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            ys[u] = p < e ? adj[p] : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            const uint32_t y = ys[u];
            if (y > x && y <= cmax) {
                uint32_t pos = (uint32_t)lower_bound_u32(C, nc, y);
                if (pos < nc && C[pos] == y) bits |= 1u << pos;
            }
        }
        if (__shfl_sync(0xffffffffu, ys[kScanChunks - 1], 31) > cmax) break;
    }
    return __reduce_or_sync(0xffffffffu, bits);
}

// Warp builds one-word rows for |C| <= 32 (rows[i] for i < nc).  The last
// candidate's row is empty (no candidate lies above it).
template <class OFF>
__device__ __forceinline__ void warp_build_rows32(const uint32_t* C, uint32_t nc,
                                                  const OFF* ne, const uint32_t* adj,
                                                  const OFF* nb, uint32_t* rows) {
    const unsigned lane = lane_id();
    if (nc == 0) return;
    const uint32_t cmax = C[nc - 1];
    for (uint32_t i = 0; i + 1 < nc; i++) {
        const uint32_t x = C[i];
        const uint32_t bits = warp_row32(C, nc, cmax, x, adj, nb[x], ne[x]);
        if (lane == 0) rows[i] = bits;
    }
    if (lane == 0) rows[nc - 1] = 0;
    __syncwarp();
}

// warp_build_rows32 (nc > 0) with the bounds of all lists loaded by a lane each
// and four lists' first entries in flight: 32 warps an SM alone do not hide the
// two dependent loads a list takes otherwise.
template <class OFF>
__device__ __forceinline__ void warp_rows32_ahead(const uint32_t* C, uint32_t nc, const OFF* ne,
                                                  const uint32_t* adj, const OFF* nb,
                                                  uint32_t* rows) {
    const unsigned full = 0xffffffffu, lane = lane_id();
    const uint32_t cmax = C[nc - 1], m = nc - 1;
    OFF lb = 0, le = 0;
    if (lane < m) {
        lb = nb[C[lane]];
        le = ne[C[lane]];
    }
    for (uint32_t i0 = 0; i0 < m; i0 += 4) {
        OFF b[4], e[4];
        uint32_t y[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t i = i0 + q < m ? i0 + q : m - 1;
            b[q] = __shfl_sync(full, lb, i);
            e[q] = __shfl_sync(full, le, i);
            y[q] = b[q] + lane < e[q] ? adj[b[q] + lane] : kNone;
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t i = i0 + q;
            if (i >= m) break;
            uint32_t bits = 0;
            for (OFF p = b[q];;) {
                if (y[q] <= cmax) {
                    const uint32_t pos = (uint32_t)lower_bound_u32(C, nc, y[q]);
                    if (pos < nc && C[pos] == y[q]) bits |= 1u << pos;
                }
                p += 32;
                if (p >= e[q] || __shfl_sync(full, y[q], 31) > cmax) break;
                y[q] = p + lane < e[q] ? adj[p + lane] : kNone;
            }
            bits = __reduce_or_sync(full, bits);
            if (lane == 0) rows[i] = bits;
        }
    }
    if (lane == 0) rows[m] = 0;
    __syncwarp();
}

// ---------------------------------------------------------------------------
// Per-candidate credits.  An r-clique listed as positions j1 < ... < jr of C
// adds one to each member's counter.  The last member of a clique is one bit
// of the leaf mask P & rows[j_{r-1}], so it is credited through bit-sliced
// counters held in registers: 32 counters of kSlices bits, counter b being
// bit b of S[0..kSlices-1] (S[0] least significant); adding a mask adds one
// to every counter whose bit is set, by ripple carry.  The counters are
// flushed (one shared-memory atomic per non-zero counter) before any of them
// can reach 2^kSlices.  The other members are credited once per search node
// with the number of cliques below it, instead of once per clique.
constexpr int kSlices = 8;
constexpr uint32_t kSliceAdds = (1u << kSlices) - 1;   // adds between flushes

struct BitSliced {
    uint32_t S[kSlices];
    uint32_t adds;
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < kSlices; i++) S[i] = 0;
        adds = 0;
    }
    __device__ __forceinline__ void add(uint32_t m) {
        uint32_t carry = m;
#pragma unroll
        for (int i = 0; i < kSlices; i++) {
            uint32_t t = S[i] & carry;
            S[i] ^= carry;
            carry = t;
            if (!carry) break;
        }
        adds++;
    }
    // cnt[b] += counter b for every b; then zero.
    template <class T>
    __device__ __forceinline__ void flush(T* cnt) {
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < kSlices; i++) any |= S[i];
        while (any) {
            int b = __ffs(any) - 1;
            any &= any - 1;
            uint32_t v = 0;
#pragma unroll
            for (int i = 0; i < kSlices; i++) v |= ((S[i] >> b) & 1u) << i;
            atomicAdd(&cnt[b], (T)v);
        }
        clear();
    }
};

// ---------------------------------------------------------------------------
// Warp DFS over one-word rows: lane i takes the cliques whose first member
// is candidate i.  Counts r-cliques (r >= 2) in G[C]; adds per-candidate
// counts into cnt[] (shared memory) and returns the warp total (all lanes).
// A node at depth d has chosen d members (sel[1..d]); P[d] holds the
// candidates adjacent to all of them.  Nodes at depth r - 2 enumerate their
// leaves in one loop.
__device__ __forceinline__ unsigned long long warp_dfs32(const uint32_t* rows, uint32_t nc,
                                                        int r, unsigned* cnt) {
    unsigned lane = lane_id();
    unsigned long long total = 0;
    if (lane < nc) {
        BitSliced bs;
        bs.clear();
        if (r == 2) {
            uint32_t last = rows[lane];
            unsigned c = __popc(last);
            if (c) {
                bs.add(last);
                atomicAdd(&cnt[lane], c);
                total = c;
            }
        } else {
            uint32_t P[kMaxDepth], rem[kMaxDepth], sel[kMaxDepth];
            unsigned acc[kMaxDepth];
            int depth = 1;
            P[1] = rows[lane];
            rem[1] = P[1];
            sel[1] = lane;
            acc[1] = 0;
            // need r - 1 more members after the first
            if (__popc(P[1]) < r - 1) depth = 0;
            while (depth >= 1) {
                if (depth == r - 2) {
                    // every j left in rem is member r-1, its leaf mask the last members
                    uint32_t rm = rem[depth], Pd = P[depth];
                    unsigned sub = 0;
                    while (rm) {
                        int j = __ffs(rm) - 1;
                        rm &= rm - 1;
                        uint32_t last = Pd & rows[j];
                        unsigned c = __popc(last);
                        if (c) {
                            bs.add(last);
                            if (bs.adds == kSliceAdds) bs.flush(cnt);
                            atomicAdd(&cnt[j], c);
                            sub += c;
                        }
                    }
                    acc[depth] += sub;
                } else if (rem[depth]) {
                    int j = __ffs(rem[depth]) - 1;
                    rem[depth] &= rem[depth] - 1;
                    uint32_t pn = P[depth] & rows[j];
                    if (__popc(pn) >= r - depth - 1) {
                        depth++;
                        sel[depth] = j;
                        P[depth] = pn;
                        rem[depth] = pn;
                        acc[depth] = 0;
                    }
                    continue;
                }
                // leave the node: credit its member with the cliques below it
                unsigned a = acc[depth];
                if (a) {
                    atomicAdd(&cnt[sel[depth]], a);
                    if (depth > 1) acc[depth - 1] += a;
                    else total = a;
                }
                depth--;
            }
        }
        bs.flush(cnt);
    }
    return warp_sum(total);
}

// ---------------------------------------------------------------------------
// Block-level bitmap routines for |C| <= 1024 candidates.
//
// Rows are symmetric (bit j of row i and bit i of row j for each edge of
// G[C]), W = ceil(nc / 32) words at a stride of Ws = row_stride(W) words.  The
// search fixes members in increasing order; a node is the set P of the
// candidates that extend them.  Its last two members are the edges of G[P]:
// a lane takes one candidate j of P and sums popc(P & row j) over the words,
// which is j's degree in G[P] -- the number of cliques j is in as either of
// the last two members -- so one addition credits it and half the sum over P
// is the number of cliques.  A lane per candidate needs no reduction, no
// leaf bit-counters and one shared atomic per candidate, where a lane per word
// needed some 25 instructions for every candidate: listing R-MAT scale 18,
// h = 5: 164 -> 43 ms, scale 17, h = 4: 7.2 -> 4.3 ms.  Bound by the row loads
// (bank conflicts between candidates' rows) and the instructions around a
// node; small sets of three members to go are searched in registers instead
// (warp_triangles_reg).
//
// The stride is 4 words times an odd number, so that the 16-byte row loads of
// eight lanes fall into different banks.
__host__ __device__ constexpr uint32_t row_stride(uint32_t W) {
    return ((W + 3u) / 4u | 1u) * 4u;
}
constexpr uint32_t kRowStrideMax = row_stride(kBitmapMax / 32);   // 36
constexpr uint32_t kWindow = 8192;                                 // see block_window
constexpr uint32_t kWindowWords = kWindow / 2;
// A warp's scratch: its node's words and the positions of its set bits.
constexpr uint32_t kLeafList = 256;
constexpr uint32_t kWarpScratch = kRowStrideMax + kLeafList / 2;  // words
// Shared words of a bitmap problem of at most bcap candidates (64-bit
// counters, candidates, rows, window, scratch of nw warps); the rows start at
// word bitmap_rows_at(bcap), the scratch at bitmap_scratch_at(bcap) and the
// window before it.
__host__ __device__ constexpr uint32_t bitmap_rows_at(uint32_t bcap) {
    return (3u * bcap + 3u) & ~3u;
}
__host__ __device__ constexpr uint32_t bitmap_words(uint32_t bcap, uint32_t nw) {
    return bitmap_rows_at(bcap) + bcap * row_stride((bcap + 31u) / 32u) + kWindowWords +
           nw * kWarpScratch;
}
__host__ __device__ constexpr uint32_t bitmap_scratch_at(uint32_t bcap) {
    return bitmap_rows_at(bcap) + bcap * row_stride((bcap + 31u) / 32u) + kWindowWords;
}

// Positions in C by id for the kWindow largest ids (16-bit, in shared memory):
// candidates crowd at the high ranks, and there a look-up replaces the ten
// dependent shared loads of a binary search.
__device__ __forceinline__ uint32_t window_base(uint32_t cmax) {
    return cmax >= kWindow ? cmax - (kWindow - 1u) : 0u;
}
// Every thread of the block calls it; the caller synchronises after it.  It
// clears the table, synchronises and enters C (win: 16-byte aligned).
__device__ __forceinline__ void block_window(const uint32_t* C, uint32_t nc, uint32_t* win) {
    for (uint32_t i = threadIdx.x; i < kWindowWords / 4; i += blockDim.x)
        reinterpret_cast<uint4*>(win)[i] = make_uint4(kNone, kNone, kNone, kNone);
    __syncthreads();
    if (nc == 0) return;
    const uint32_t w0 = window_base(C[nc - 1]);
    for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x)
        if (C[i] >= w0) reinterpret_cast<uint16_t*>(win)[C[i] - w0] = (uint16_t)i;
}
// The position of y <= cmax in C, or kNone.
__device__ __forceinline__ uint32_t find_pos(const uint32_t* C, uint32_t nc, const uint32_t* win,
                                             uint32_t w0, uint32_t y) {
    if (y >= w0) {
        const uint32_t p = reinterpret_cast<const uint16_t*>(win)[y - w0];
        return p == 0xffffu ? kNone : p;
    }
    const uint32_t p = (uint32_t)lower_bound_u32(C, nc, y);
    return p < nc && C[p] == y ? p : kNone;
}

// Hits of adj[b, e) in C as scan_row_hits, found through the window: cnt[2 pos]
// += 1 (the low words of 64-bit counters).
__device__ __forceinline__ unsigned scan_row_window(const uint32_t* C, uint32_t nc, uint32_t cmax,
                                                    const uint32_t* win, uint32_t w0,
                                                    const uint32_t* adj, uint64_t b, uint64_t e,
                                                    unsigned* cnt) {
    const unsigned lane = lane_id();
    unsigned hits = 0;
    for (uint64_t p0 = b; p0 < e; p0 += 32 * kScanChunks) {
        uint32_t ys[kScanChunks];
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            ys[u] = p < e ? adj[p] : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < kScanChunks; u++) {
            if (ys[u] <= cmax) {
                const uint32_t pos = find_pos(C, nc, win, w0, ys[u]);
                if (pos != kNone) {
                    atomicAdd(&cnt[2 * pos], 1u);
                    hits++;
                }
            }
        }
        if (__shfl_sync(0xffffffffu, ys[kScanChunks - 1], 31) > cmax) break;
    }
    return hits;
}

// rows: nc * row_stride(W) words, zeroed by the caller; win: C's window
// (block_window).  num (may be null): the row number of each candidate.
template <class OFF>
__device__ __forceinline__ void block_build_rows(const uint32_t* C, uint32_t nc, uint32_t W,
                                                 const OFF* ne, const uint32_t* adj,
                                                 const OFF* nb, uint32_t* rows,
                                                 const uint32_t* win,
                                                 const uint16_t* num = nullptr) {
    const unsigned lane = lane_id();
    const unsigned nw = blockDim.x >> 5;
    if (nc == 0) return;
    const uint32_t Ws = row_stride(W);
    const uint32_t cmax = C[nc - 1], w0 = window_base(cmax);
    for (uint32_t i = warp_id(); i + 1 < nc; i += nw) {
        const uint32_t x = C[i];
        const uint64_t b = nb[x], e = ne[x];
        for (uint64_t p0 = b; p0 < e; p0 += 32 * kScanChunks) {
            uint32_t ys[kScanChunks];
#pragma unroll
            for (int u = 0; u < kScanChunks; u++) {
                uint64_t p = p0 + u * 32 + lane;
                ys[u] = p < e ? adj[p] : 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < kScanChunks; u++) {
                const uint32_t y = ys[u];
                if (y > x && y <= cmax) {
                    const uint32_t pos = find_pos(C, nc, win, w0, y);
                    if (pos != kNone) {
                        const uint32_t a = num ? num[i] : i, c = num ? num[pos] : pos;
                        atomicOr(&rows[a * Ws + (c >> 5)], 1u << (c & 31));
                        atomicOr(&rows[c * Ws + (a >> 5)], 1u << (a & 31));
                    }
                }
            }
            if (__shfl_sync(0xffffffffu, ys[kScanChunks - 1], 31) > cmax) break;
        }
    }
}

// A bitmap problem as one warp sees it.  small: no counter passes 2^32 - 1
// (r <= 4 members of at most 1024), so that 32-bit shared atomics on the low
// word of a 64-bit counter do.
struct BitmapWarp {
    const uint32_t* rows;
    uint32_t W, Ws;
    unsigned long long* cnt;
    uint32_t* sP;          // [Ws]
    uint16_t* list;        // [kLeafList]
    bool small;
    uint32_t nd;           // only candidates below nd are credited
    __device__ __forceinline__ void credit(uint32_t j, unsigned long long v) const {
        if (j >= nd) return;
        if (small) atomicAdd(reinterpret_cast<unsigned*>(cnt + j), (unsigned)v);
        else atomicAdd(cnt + j, v);
    }
    __device__ __forceinline__ uint32_t row_word(uint32_t j) const {
        const unsigned l = lane_id();
        return l < W ? rows[j * Ws + l] : 0u;
    }
};

// Bitwise ones + x + y: ones takes the sums' low bits, the carries are returned
// (a full adder a bit).  Two words then cost one popc and two three-input
// logic operations, which run at four times the rate, instead of two popc.
__device__ __forceinline__ uint32_t carry_add(uint32_t& ones, uint32_t x, uint32_t y) {
    const uint32_t c = (ones & x) | (ones & y) | (x & y);
    ones ^= x ^ y;
    return c;
}

// The positions base .. base + kLeafList - 1 among P's set bits into B.list
// (pc, inc: bits of this lane's word and of the words up to it).
__device__ __forceinline__ void warp_list(const BitmapWarp& B, uint32_t Pw, uint32_t pc,
                                          uint32_t inc, uint32_t base) {
    uint32_t at = inc - pc, w = Pw;
    while (w) {
        const uint32_t b = __ffs(w) - 1u;
        w &= w - 1u;
        if (at >= base && at < base + kLeafList)
            B.list[at - base] = (uint16_t)(lane_id() * 32 + b);
        at++;
    }
    __syncwarp();
}
__device__ __forceinline__ uint32_t warp_incl_sum(uint32_t x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane_id() >= o) x += y;
    }
    return x;
}

// Edges of G[P] (this lane's word of P given; all lanes get the result); each
// end is credited with its degree.
__device__ __forceinline__ unsigned long long warp_edges(const BitmapWarp& B, uint32_t Pw) {
    const unsigned full = 0xffffffffu, lane = lane_id();
    const unsigned nz = __ballot_sync(full, Pw != 0);
    if (!nz) return 0;
    const uint32_t lo = (uint32_t)(__ffs(nz) - 1) >> 2, hi = ((31u - __clz(nz)) >> 2) + 1u;
    const uint32_t pc = __popc(Pw);
    const uint32_t inc = warp_incl_sum(pc);
    const uint32_t total = __shfl_sync(full, inc, 31);
    if (total < 2) return 0;
    if (lane < B.Ws) B.sP[lane] = Pw;
    unsigned sum = 0;
    for (uint32_t base = 0; base < total; base += kLeafList) {
        warp_list(B, Pw, pc, inc, base);
        const uint32_t m = total - base < kLeafList ? total - base : kLeafList;
        for (uint32_t q = lane; q < m; q += 32) {
            const uint32_t j = B.list[q];
            const uint4* row = reinterpret_cast<const uint4*>(B.rows + j * B.Ws);
            const uint4* P4 = reinterpret_cast<const uint4*>(B.sP);
            unsigned twos = 0, ones = 0;
            for (uint32_t v = lo; v < hi; v++) {
                const uint4 a = row[v], p = P4[v];
                twos += __popc(carry_add(ones, a.x & p.x, a.y & p.y));
                twos += __popc(carry_add(ones, a.z & p.z, a.w & p.w));
            }
            const unsigned s = 2 * twos + __popc(ones);
            if (s) B.credit(j, s);
            sum += s;
        }
        __syncwarp();
    }
    return __reduce_add_sync(full, sum) >> 1;   // sum <= 1024 * 1023
}

// Triangles of G[P] for p members of P, 32 (K - 1) < p <= 32 K, their positions
// in B.list: G[P] is gathered into registers, a lane holding the rows of K
// members over the members only, so that a node of the search (the members
// above j adjacent to it) takes no shared memory at all: K broadcasts and at
// most K * K popc.  In the shared rows a node costs its list, its row loads
// over the whole width of G[C] (with bank conflicts) and its credits, some 570
// issue slots on R-MAT scale 18 (h = 5, 27 candidates a node).  That listing
// call: 49.9 -> 24.7 ms.  Bound by instruction issue (77 % of the slots; popc
// takes 22 % of its pipe).
template <int K>
__device__ unsigned warp_triangles_reg(const BitmapWarp& B, uint32_t p) {
    const unsigned full = 0xffffffffu, lane = lane_id();
    uint32_t pos[K], row[K][K], cnt[K];
    const uint32_t last = p & 31u ? (1u << (p & 31u)) - 1u : full;   // members of the last 32
#pragma unroll
    for (int s = 0; s < K; s++) {
        pos[s] = s * 32 + lane < p ? B.list[s * 32 + lane] : 0u;
        cnt[s] = 0;
    }
#pragma unroll
    for (int s = 0; s < K; s++) {
#pragma unroll
        for (int w = 0; w < K; w++) row[s][w] = 0;
        const uint32_t na = p - s * 32 < 32u ? p - s * 32 : 32u;
        for (uint32_t a = 0; a < na; a++) {
            const uint32_t* r = B.rows + __shfl_sync(full, pos[s], a) * B.Ws;
#pragma unroll
            for (int w = 0; w < K; w++) {
                unsigned m = __ballot_sync(full, (r[pos[w] >> 5] >> (pos[w] & 31u)) & 1u);
                if (w == K - 1) m &= last;
                if (lane == a) row[s][w] = m;
            }
        }
    }
    unsigned total = 0;
#pragma unroll
    for (int s = 0; s < K; s++) {
        const uint32_t na = p - s * 32 < 32u ? p - s * 32 : 32u;
        for (uint32_t a = 0; a < na; a++) {
            uint32_t pn[K], any = 0;
#pragma unroll
            for (int w = s; w < K; w++) {
                pn[w] = __shfl_sync(full, row[s][w], a);
                if (w == s) pn[w] &= 0xfffffffeu << a;
                any |= pn[w];
            }
            if (!any) continue;
            unsigned sum = 0;
#pragma unroll
            for (int q = s; q < K; q++) {
                unsigned c = 0;
#pragma unroll
                for (int w = s; w < K; w++) c += __popc(row[q][w] & pn[w]);
                if (!((pn[q] >> lane) & 1u)) c = 0;
                cnt[q] += c;
                sum += c;
            }
            sum = __reduce_add_sync(full, sum) >> 1;
            if (lane == a) cnt[s] += sum;
            total += sum;
        }
    }
#pragma unroll
    for (int s = 0; s < K; s++)
        if (s * 32 + lane < p && cnt[s]) B.credit(pos[s], cnt[s]);
    __syncwarp();   // B.list is used again
    return total;
}
// P above this is searched in the shared rows: K = 5 needs 25 registers of rows
// alone, of the 64 that a block of 1,024 threads has a thread.
constexpr uint32_t kRegMembers = 32 * 4;

// RR-cliques of G[P], RR >= 2; each member is credited with those it is in.
// REG: triangles of at most kRegMembers members in registers (for callers with
// the registers to spare: r >= 4).
template <int RR, bool REG>
__device__ unsigned long long warp_cliques(const BitmapWarp& B, uint32_t Pw) {
    if constexpr (RR == 2) {
        return warp_edges(B, Pw);
    } else {
        const unsigned full = 0xffffffffu, lane = lane_id();
        if constexpr (RR == 3 && REG) {
            const uint32_t pc = __popc(Pw);
            const uint32_t p = __reduce_add_sync(full, pc);
            if (p < 3) return 0;
            if (p <= kRegMembers) {
                warp_list(B, Pw, pc, warp_incl_sum(pc), 0);
                if (p <= 32) return warp_triangles_reg<1>(B, p);
                if (p <= 64) return warp_triangles_reg<2>(B, p);
                if (p <= 96) return warp_triangles_reg<3>(B, p);
                return warp_triangles_reg<4>(B, p);
            }
        }
        unsigned long long acc = 0;
        uint32_t rem = Pw;
        for (;;) {
            const unsigned have = __ballot_sync(full, rem != 0);
            if (!have) break;
            const int fl = __ffs(have) - 1;
            const uint32_t b = __ffs(__shfl_sync(full, rem, fl)) - 1u;
            if ((int)lane == fl) rem &= rem - 1;
            const uint32_t j = (uint32_t)fl * 32 + b;
            // rem holds exactly the members of P above j
            const uint32_t pn = rem & B.row_word(j);
            unsigned long long sub;
            if constexpr (RR == 3) {
                sub = warp_edges(B, pn);
            } else {
                if (__reduce_add_sync(full, (unsigned)__popc(pn)) < RR - 1) continue;
                sub = warp_cliques<RR - 1, REG>(B, pn);
            }
            if (sub) {
                if (lane == 0) B.credit(j, sub);
                acc += sub;
            }
        }
        return acc;
    }
}

template <bool REG>
__device__ __forceinline__ unsigned long long warp_cliques_of(const BitmapWarp& B, uint32_t Pw,
                                                             int rr) {
    switch (rr) {
        case 2: return warp_cliques<2, REG>(B, Pw);
        case 3: return warp_cliques<3, REG>(B, Pw);
        case 4: return warp_cliques<4, REG>(B, Pw);
        case 5: return warp_cliques<5, REG>(B, Pw);
        default: return warp_cliques<6, REG>(B, Pw);   // r <= DSD_MAX_H - 1 = 7
    }
}

__device__ __forceinline__ BitmapWarp bitmap_warp(const uint32_t* rows, uint32_t W, int r,
                                                  unsigned long long* cnt, uint32_t* scratch,
                                                  uint32_t nd) {
    BitmapWarp B;
    B.rows = rows;
    B.W = W;
    B.Ws = row_stride(W);
    B.cnt = cnt;
    B.sP = scratch + warp_id() * kWarpScratch;
    B.list = reinterpret_cast<uint16_t*>(B.sP + kRowStrideMax);
    B.small = r <= 4;
    B.nd = nd;
    // words past the lanes' 32 (a full-width stride) stay zero
    if (lane_id() < kRowStrideMax - 32) B.sP[32 + lane_id()] = 0;
    __syncwarp();
    return B;
}

// r-cliques of G[C], r >= 2, with every member's count added to cnt (zeroed
// by the caller).  Warps take first members i from the shared counter *next_i
// (zero on entry; the early candidates, with the largest searches above them,
// go first); r >= 3: only those of start, start + step, ... below nd, and
// only candidates below nd are credited.  scratch: kWarpScratch words a warp, 16-byte aligned.  Returns this
// thread's share of the total (sum over the block = total).
template <bool REG = false>
__device__ __forceinline__ unsigned long long block_dfs(const uint32_t* rows, uint32_t nc,
                                                       uint32_t W, int r,
                                                       unsigned long long* cnt,
                                                       uint32_t* next_i, uint32_t* scratch,
                                                       uint32_t start = 0, uint32_t step = 1,
                                                       uint32_t nd = kNone) {
    const unsigned full = 0xffffffffu, lane = lane_id();
    unsigned long long total = 0;
    if (r == 2) {
        // edges: a candidate's count is its degree
        const uint32_t Ws = row_stride(W);
        for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
            unsigned s = 0, below = 0;
            for (uint32_t w = 0; w < W; w++) {
                const uint32_t x = rows[i * Ws + w];
                s += __popc(x);
                below += w < (i >> 5) ? __popc(x)
                                      : (w == (i >> 5) ? __popc(x & ((1u << (i & 31u)) - 1u)) : 0);
            }
            cnt[i] += s;
            total += below;
        }
        return total;
    }
    if (nd > nc) nd = nc;
    const BitmapWarp B = bitmap_warp(rows, W, r, cnt, scratch, nd);
    for (;;) {
        uint32_t i = 0;
        if (lane == 0) i = atomicAdd(next_i, 1u);
        i = start + step * __shfl_sync(full, i, 0);
        if (i >= nd) break;
        uint32_t P = B.row_word(i);
        const uint32_t iw = i >> 5;
        if (lane < iw) P = 0;
        else if (lane == iw) P &= (i & 31u) == 31u ? 0u : 0xffffffffu << ((i & 31u) + 1u);
        if ((int)__reduce_add_sync(full, (unsigned)__popc(P)) < r - 1) continue;
        const unsigned long long c = warp_cliques_of<REG>(B, P, r - 1);
        if (c) {
            if (lane == 0) B.credit(i, c);
            total += c;
        }
    }
    return lane == 0 ? total : 0ull;
}

}  // namespace dsd
