// Many small graphs (mixed h) in one persistent launch.
//
// Each CTA takes graphs from an atomic work queue (largest first) and runs
// the whole path of one graph by itself -- CSR build (Sec. 2 data model),
// degeneracy peel (edge k-cores, Def. 5), rank relabelling, h-clique
// clique-degrees (Def. 3) and the level-synchronous (k,Psi)-core peel
// (Algorithm 3) with its level statistics, then the CoreApp outputs (k_max
// core, Lemma 6; densest level, Pruning1).  Within a graph the phases are
// separated by __syncthreads only: no grid barrier, no host round trip.
// Per-graph scratch is a private slice of one workspace per CTA.
//
// Graph size limits: n <= 65535 vertices (a vertex's round and id share a
// 32-bit key, and long rows are sorted by 16 bits) and, for h = 3 and 4, at
// most 512 higher-ranked neighbours per vertex.
#include "cliques.cuh"
#include "graph.cuh"

#include <string.h>

namespace dsd {
namespace {

constexpr uint32_t kBatchMaxN = 65535;
constexpr uint32_t kBatchMaxDplus = 512;
enum : uint32_t { kBOk = 0, kBInvalid = 1, kBUnsupported = 2 };
enum : uint32_t { kAl = 0, kFr = 1, kGo = 2 };

struct BatchDesc {
    uint64_t e_off;     // first edge of this graph in src/dst
    uint64_t core_off;  // first entry of its core numbers (~0: not wanted)
    uint32_t m;         // raw edges
    uint32_t n;
    int32_t h;
    uint32_t pad;
};

struct BatchRes {
    unsigned long long kmax, kmax_core_mu, best_k, densest_mu, mu, m_clean;
    uint32_t kmax_core_size, densest_size, nlevels, status;
};

// Per-CTA workspace (global memory), sized for the largest graph.
struct Work {
    uint32_t* k1;       // rows being built / scratch, max(E, n)
    uint32_t* k2;       // scratch; (round, id) keys of the vertices, max(E, n)
    uint32_t* adj;      // rows (caller ids), E
    uint32_t* radj;     // rows (ranks), E
    uint32_t* off;      // n + 1
    uint32_t* roff;     // n + 1
    uint32_t* rsplit;   // n
    uint32_t* rnd;      // n
    uint32_t* new_of;   // n
    uint32_t* old_of;   // n
    uint32_t* st;       // n
    uint32_t* fa;       // n  (frontier)
    uint32_t* fb;       // n  (next frontier)
    uint32_t* alive;    // n
    unsigned long long* deg;   // n
    unsigned long long* core;  // n
    unsigned long long* lk;    // n + 1
    unsigned long long* lm;    // n + 1
    uint32_t* ls;              // n + 1
};

struct BatchArgs {
    const BatchDesc* desc;
    const uint32_t* order;     // graphs, largest first
    uint32_t count;
    const uint32_t* src;
    const uint32_t* dst;
    BatchRes* res;
    unsigned long long* cores; // concatenated core numbers (may be null)
    uint32_t* queue;           // work counter
    uint8_t* ws;               // workspaces
    uint64_t ws_stride;        // bytes per CTA
    uint32_t maxn;
    uint64_t maxe;
};

__device__ __forceinline__ uint8_t* align_up(uint8_t* p) {
    return (uint8_t*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
}

__device__ Work carve(uint8_t* base, uint32_t maxn, uint64_t maxe) {
    Work w;
    uint8_t* p = align_up(base);
    auto take = [&](size_t bytes) {
        uint8_t* r = p;
        p = align_up(p + bytes);
        return r;
    };
    const uint64_t keys = maxe > maxn ? maxe : (uint64_t)maxn;   // an entry, or a vertex
    w.k1 = (uint32_t*)take(keys * 4);
    w.k2 = (uint32_t*)take(keys * 4);
    w.adj = (uint32_t*)take(maxe * 4);
    w.radj = (uint32_t*)take(maxe * 4);
    w.off = (uint32_t*)take(((size_t)maxn + 1) * 4);
    w.roff = (uint32_t*)take(((size_t)maxn + 1) * 4);
    w.rsplit = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.rnd = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.new_of = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.old_of = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.st = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.fa = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.fb = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.alive = (uint32_t*)take((size_t)maxn * 4 + 4);
    w.deg = (unsigned long long*)take((size_t)maxn * 8 + 8);
    w.core = (unsigned long long*)take((size_t)maxn * 8 + 8);
    w.lk = (unsigned long long*)take(((size_t)maxn + 1) * 8);
    w.lm = (unsigned long long*)take(((size_t)maxn + 1) * 8);
    w.ls = (uint32_t*)take(((size_t)maxn + 1) * 4);
    return w;
}

// Shared-memory layout used by the phases (they run one after another).
template <int NT>
struct Smem {
    static constexpr int NW = NT / 32;
    uint32_t wcnt[NW][256];     // radix: per-warp digit counts
    uint32_t base[256];         // radix: digit offsets
    uint32_t tcnt[256];
    uint32_t wbuf[NW][2 * kBatchMaxDplus + 64];   // per-warp candidate lists
    unsigned long long red[NW];
    uint32_t ured[NW];
    uint32_t cnt1, cnt2, flag;
    unsigned long long k, mu_alive;
};

// ------------------------------------------------ block-level building blocks

// Exclusive prefix of per-thread counts; returns this thread's prefix and the
// total (all threads).
template <int NT>
__device__ __forceinline__ uint32_t bscan(uint32_t v, uint32_t* ured, uint32_t* total) {
    unsigned lane = lane_id(), wid = warp_id();
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane >= o) x += y;
    }
    if (lane == 31) ured[wid] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int w = 0; w < NT / 32; w++) {
        uint32_t t = ured[w];
        before += (w < (int)wid) ? t : 0u;
        all += t;
    }
    __syncthreads();
    *total = all;
    return before + x - v;
}

template <int NT>
__device__ __forceinline__ unsigned long long bmin(unsigned long long v, unsigned long long* red) {
    v = warp_min_u64(v);
    if (lane_id() == 0) red[warp_id()] = v;
    __syncthreads();
    unsigned long long m = ~0ull;
    for (int w = 0; w < NT / 32; w++) m = red[w] < m ? red[w] : m;
    __syncthreads();
    return m;
}

template <int NT>
__device__ __forceinline__ unsigned long long bsum(unsigned long long v, unsigned long long* red) {
    v = warp_sum(v);
    if (lane_id() == 0) red[warp_id()] = v;
    __syncthreads();
    unsigned long long m = 0;
    for (int w = 0; w < NT / 32; w++) m += red[w];
    __syncthreads();
    return m;
}

// Stable LSD radix sort of a[0..cnt) (u32 keys below 2^bits) by one CTA; the
// result ends in a (b is scratch).  Digits of 8 bits; each warp ranks its
// keys in order with match masks, so equal digits keep their order.
template <int NT>
__device__ void block_radix_sort(uint32_t* a, uint32_t* b, uint32_t cnt, int bits, Smem<NT>& S) {
    constexpr int NW = NT / 32;
    constexpr int ITEMS = 8;
    constexpr uint32_t TILE = NT * ITEMS;
    const unsigned lane = lane_id(), wid = warp_id();
    uint32_t* src = a;
    uint32_t* dst = b;
    int passes = 0;
    for (int shift = 0; shift < bits; shift += 8) {
        // digit histogram of the whole array -> exclusive offsets
        for (uint32_t i = threadIdx.x; i < 256; i += NT) S.base[i] = 0;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < cnt; i += NT) atomicAdd(&S.base[(src[i] >> shift) & 255u], 1u);
        __syncthreads();
        {
            uint32_t all;
            const uint32_t ex =
                bscan<NT>(threadIdx.x < 256 ? S.base[threadIdx.x] : 0u, S.ured, &all);
            if (threadIdx.x < 256) S.base[threadIdx.x] = ex;
        }
        __syncthreads();
        for (uint32_t t0 = 0; t0 < cnt; t0 += TILE) {
            for (uint32_t i = threadIdx.x; i < NW * 256; i += NT) (&S.wcnt[0][0])[i] = 0;
            __syncthreads();
            uint32_t key[ITEMS], rk[ITEMS];
            // warp w holds tile entries [w*32*ITEMS, (w+1)*32*ITEMS), item j at j*32 + lane
#pragma unroll
            for (int j = 0; j < ITEMS; j++) {
                uint32_t idx = t0 + wid * 32 * ITEMS + j * 32 + lane;
                bool ok = idx < cnt;
                key[j] = ok ? src[idx] : 0u;
                uint32_t d = ok ? ((key[j] >> shift) & 255u) : 256u;
                unsigned peers = __match_any_sync(0xffffffffu, d);
                uint32_t before = 0;
                if (ok) {
                    int leader = __ffs(peers) - 1;
                    uint32_t prior = 0;
                    if ((int)lane == leader) prior = S.wcnt[wid][d];
                    prior = __shfl_sync(peers, prior, leader);
                    before = prior + __popc(peers & ((1u << lane) - 1u));
                    if ((int)lane == leader) S.wcnt[wid][d] = prior + __popc(peers);
                }
                rk[j] = before;
                __syncwarp();
            }
            __syncthreads();
            // per digit: prefix over warps, tile total
            for (uint32_t d = threadIdx.x; d < 256; d += NT) {
                uint32_t run = 0;
                for (int w = 0; w < NW; w++) {
                    uint32_t t = S.wcnt[w][d];
                    S.wcnt[w][d] = run;
                    run += t;
                }
                S.tcnt[d] = run;
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < ITEMS; j++) {
                uint32_t idx = t0 + wid * 32 * ITEMS + j * 32 + lane;
                if (idx < cnt) {
                    uint32_t d = (key[j] >> shift) & 255u;
                    dst[S.base[d] + S.wcnt[wid][d] + rk[j]] = key[j];
                }
            }
            __syncthreads();
            for (uint32_t d = threadIdx.x; d < 256; d += NT) S.base[d] += S.tcnt[d];
            __syncthreads();
        }
        uint32_t* t = src;
        src = dst;
        dst = t;
        passes++;
    }
    if (passes & 1)
        for (uint32_t i = threadIdx.x; i < cnt; i += NT) a[i] = src[i];
    __syncthreads();
}

// Exclusive prefix sums of a[0..n) into out[0..n] by one CTA; returns the total.
template <int NT>
__device__ uint32_t block_prefix(const uint32_t* a, uint32_t n, uint32_t* out, Smem<NT>& S) {
    uint32_t run = 0;
    for (uint32_t t0 = 0; t0 < n; t0 += NT) {
        const uint32_t i = t0 + threadIdx.x;
        uint32_t tot;
        const uint32_t ex = bscan<NT>(i < n ? a[i] : 0u, S.ured, &tot);
        if (i < n) out[i] = run + ex;
        run += tot;
    }
    if (threadIdx.x == 0) out[n] = run;
    __syncthreads();
    return run;
}

// Sorts the rows vals[pos[v] .. pos[v] + len[v]) ascending in place, dropping
// repeats; len[v] becomes the unique length.  A warp a row: a bitonic network
// in registers up to 32 entries, in its own buffer up to kWarpSortMax; longer
// rows (listed in `longs`) by the whole CTA.  One radix sort over all (row,
// entry) keys took 8 passes over the edges and block barriers for each tile:
// the largest graph of a batch (50,000 vertices, 546,000 edges, h = 4) spent
// some 18 of 46 ms there.
constexpr uint32_t kWarpSortMax = 512;
template <int NT>
__device__ void block_sort_rows(uint32_t* vals, uint32_t* scratch, const uint32_t* pos,
                                uint32_t* len, uint32_t n, uint32_t* longs, Smem<NT>& S) {
    constexpr int NW = NT / 32;
    const unsigned lane = lane_id(), wid = warp_id();
    if (threadIdx.x == 0) S.cnt2 = 0;
    __syncthreads();
    uint32_t* sw = S.wbuf[wid];
    for (uint32_t v = wid; v < n; v += NW) {
        const uint32_t l = len[v];
        uint32_t* row = vals + pos[v];
        if (l <= 32) {
            uint32_t x = lane < l ? row[lane] : kNone;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
                    const bool asc = (lane & k) == 0, lower = (lane & j) == 0;
                    x = (lower == asc) ? min(x, y) : max(x, y);
                }
            }
            const uint32_t prev = __shfl_up_sync(0xffffffffu, x, 1);
            const bool keep = lane < l && (lane == 0 || x != prev);
            const unsigned b = __ballot_sync(0xffffffffu, keep);
            if (keep) row[__popc(b & ((1u << lane) - 1u))] = x;
            if (lane == 0) len[v] = __popc(b);
            continue;
        }
        if (l > kWarpSortMax) {
            if (lane == 0) longs[atomicAdd(&S.cnt2, 1u)] = v;
            continue;
        }
        uint32_t N = 64;
        while (N < l) N <<= 1;
        for (uint32_t j = lane; j < N; j += 32) sw[j] = j < l ? row[j] : kNone;
        __syncwarp();
        for (uint32_t k = 2; k <= N; k <<= 1) {
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t x = lane; x < N; x += 32) {
                    const uint32_t y = x ^ j;
                    if (y > x) {
                        const bool asc = (x & k) == 0;
                        const uint32_t a = sw[x], b = sw[y];
                        if ((a > b) == asc) {
                            sw[x] = b;
                            sw[y] = a;
                        }
                    }
                }
                __syncwarp();
            }
        }
        uint32_t out = 0;
        for (uint32_t b0 = 0; b0 < l; b0 += 32) {
            const uint32_t x = b0 + lane;
            const uint32_t val = x < l ? sw[x] : 0u;
            const bool keep = x < l && (x == 0 || val != sw[x - 1]);
            const unsigned bal = __ballot_sync(0xffffffffu, keep);
            if (keep) row[out + __popc(bal & ((1u << lane) - 1u))] = val;
            out += __popc(bal);
        }
        if (lane == 0) len[v] = out;
        __syncwarp();
    }
    __syncthreads();
    const uint32_t nl = S.cnt2;
    for (uint32_t i = 0; i < nl; i++) {
        const uint32_t v = longs[i], l = len[v];
        uint32_t* row = vals + pos[v];
        block_radix_sort<NT>(row, scratch, l, 16, S);   // ids below 2^16
        uint32_t out = 0;
        for (uint32_t t0 = 0; t0 < l; t0 += NT) {
            const uint32_t x = t0 + threadIdx.x;
            const uint32_t val = x < l ? row[x] : 0u;
            const bool keep = x < l && (x == 0 || row[x - 1] != val);
            uint32_t tot;
            const uint32_t at = bscan<NT>(keep ? 1u : 0u, S.ured, &tot);
            if (keep) scratch[out + at] = val;
            out += tot;
        }
        __syncthreads();
        for (uint32_t x = threadIdx.x; x < out; x += NT) row[x] = scratch[x];
        if (threadIdx.x == 0) len[v] = out;
        __syncthreads();
    }
}

// ------------------------------------------------------------ peeling

struct BPeel {
    const uint32_t* off;
    const uint32_t* adj;
    const uint32_t* nplus;   // start of N+ per vertex (h >= 3)
    uint32_t n;
    int h;
    unsigned long long* deg;
    unsigned long long* core;
    uint32_t* rnd;           // may be null
    uint32_t* st;
    uint32_t* alive;
    uint32_t* fa;
    uint32_t* fb;
    uint32_t* tmp;           // n words
    unsigned long long* lk;
    unsigned long long* lm;
    uint32_t* ls;
    unsigned long long mu0;
};

__device__ __forceinline__ bool bcand(const BPeel& B, uint32_t x, uint32_t v) {
    uint32_t s = B.st[x];
    return s == kAl || (s == kFr && x > v);
}

__device__ __forceinline__ void bdec(const BPeel& B, uint32_t u, unsigned long long c,
                                     unsigned long long k, uint32_t* next, uint32_t* ncnt) {
    unsigned long long old = atomic_sub_u64(&B.deg[u], c);
    if (old > k && old - c <= k) next[atomicAdd(ncnt, 1u)] = u;
}

// Lanes of this lane's group when a warp scans 32 / LPR rows at once, LPR
// lanes each (the intersection tile the launch was tuned with).
template <int LPR>
__device__ __forceinline__ unsigned group_mask() {
    if (LPR == 32) return 0xffffffffu;
    return ((1u << LPR) - 1u) << (lane_id() & ~(unsigned)(LPR - 1));
}

// (v, w) item for h >= 3, one warp: the cliques {v, w, ...} whose other
// members are candidates of v and whose smallest such member is w.
template <int LPR>
__device__ unsigned long long bitem(const BPeel& B, uint32_t v, uint32_t w, unsigned long long k,
                                    uint32_t* next, uint32_t* ncnt, uint32_t* C, uint32_t* cnt) {
    unsigned lane = lane_id();
    if (!bcand(B, w, v)) return 0;
    const uint32_t* Nv = B.adj + B.off[v];
    uint32_t dv = B.off[v + 1] - B.off[v];
    uint32_t b = B.nplus[w], e = B.off[w + 1];
    uint32_t nc = 0;
    for (uint32_t p0 = b; p0 < e; p0 += 32) {
        uint32_t p = p0 + lane;
        bool ok = false;
        uint32_t x = 0;
        if (p < e) {
            x = B.adj[p];
            if (bcand(B, x, v)) {
                uint32_t pos = (uint32_t)lower_bound_u32(Nv, dv, x);
                ok = pos < dv && Nv[pos] == x;
            }
        }
        unsigned bal = __ballot_sync(0xffffffffu, ok);
        if (ok) C[nc + __popc(bal & ((1u << lane) - 1u))] = x;
        nc += __popc(bal);
    }
    __syncwarp();
    unsigned long long tot = 0;
    if (B.h == 3) {
        tot = nc;
        for (uint32_t i = lane; i < nc; i += 32)
            if (B.st[C[i]] == kAl) bdec(B, C[i], 1ull, k, next, ncnt);
    } else {
        // h = 4: edges of G[C]; the warp scans 32 / LPR rows at once
        for (uint32_t i = lane; i < nc; i += 32) cnt[i] = 0;
        __syncwarp();
        const unsigned gl = lane & (LPR - 1), gm = group_mask<LPR>();
        unsigned long long mine = 0;
        for (uint32_t i = lane / LPR; i < nc; i += 32 / LPR) {
            uint32_t x = C[i];
            unsigned hits = 0;
            for (uint32_t p = B.nplus[x] + gl; p < B.off[x + 1]; p += LPR) {
                uint32_t y = B.adj[p];
                uint32_t pos = (uint32_t)lower_bound_u32(C, nc, y);
                if (pos < nc && C[pos] == y) { atomicAdd(&cnt[pos], 1u); hits++; }
            }
            hits = __reduce_add_sync(gm, hits);
            if (gl == 0 && hits) atomicAdd(&cnt[i], hits);
            if (gl == 0) mine += hits;
        }
        __syncwarp();
        tot = warp_sum(mine);
        if (tot)
            for (uint32_t i = lane; i < nc; i += 32)
                if (cnt[i] && B.st[C[i]] == kAl) bdec(B, C[i], cnt[i], k, next, ncnt);
        __syncwarp();
    }
    if (tot && lane == 0 && B.st[w] == kAl) bdec(B, w, tot, k, next, ncnt);
    return tot;
}

// Rows above this are shared by the block's warps in any round.
constexpr uint32_t kBatchSharedRow = 128;

// Level-synchronous peel of one graph by one CTA; returns k_max and writes
// the level records; *nl receives their number.
template <int NT, int LPR>
__device__ unsigned long long block_peel(const BPeel& B, Smem<NT>& S, uint32_t* nl) {
    constexpr int NW = NT / 32;
    const unsigned lane = lane_id(), wid = warp_id();
    uint32_t n = B.n;
    for (uint32_t v = threadIdx.x; v < n; v += NT) {
        B.st[v] = kAl;
        B.alive[v] = v;
    }
    if (threadIdx.x == 0) {
        S.cnt1 = 0;   // current frontier size
        S.mu_alive = B.mu0;
    }
    __syncthreads();
    unsigned long long k = 0;
    uint32_t na = n, left = n, nlev = 0, r = 0;   // list entries, alive vertices
    uint32_t* F = B.fa;
    uint32_t* G = B.fb;
    uint32_t nf = 0;
    for (;;) {
        if (nf == 0) {
            // level jump: minimum count and frontier; the alive list is
            // compacted when it has halved (a block scan per NT entries,
            // several barriers each; a plain pass needs none)
            unsigned long long mn = ~0ull;
            if (2 * left <= na) {
                if (threadIdx.x == 0) S.cnt2 = 0;
                __syncthreads();
                for (uint32_t t0 = 0; t0 < na; t0 += NT) {
                    uint32_t i = t0 + threadIdx.x;
                    uint32_t v = i < na ? B.alive[i] : 0u;
                    bool keep = i < na && B.st[v] == kAl;
                    uint32_t tot;
                    uint32_t at = bscan<NT>(keep ? 1u : 0u, S.ured, &tot);
                    uint32_t o = S.cnt2;
                    __syncthreads();
                    if (keep) B.alive[o + at] = v;
                    __syncthreads();
                    if (threadIdx.x == 0) S.cnt2 = o + tot;
                    __syncthreads();
                }
                na = left;
            }
            if (left == 0) break;
            for (uint32_t i = threadIdx.x; i < na; i += NT) {
                const uint32_t v = B.alive[i];
                if (B.st[v] == kAl) mn = B.deg[v] < mn ? B.deg[v] : mn;
            }
            mn = bmin<NT>(mn, S.red);
            k = mn > k ? mn : k;
            if (threadIdx.x == 0) {
                B.lk[nlev] = k;
                B.ls[nlev] = left;
                B.lm[nlev] = S.mu_alive;
                S.cnt1 = 0;
            }
            nlev++;
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < na; i += NT) {
                uint32_t v = B.alive[i];
                if (B.st[v] == kAl && B.deg[v] <= k) F[atomicAdd(&S.cnt1, 1u)] = v;
            }
            __syncthreads();
            nf = S.cnt1;
        }
        for (uint32_t i = threadIdx.x; i < nf; i += NT) B.st[F[i]] = kFr;
        if (threadIdx.x == 0) {
            S.cnt2 = 0;   // next frontier size
            S.flag = 0;   // listed rows
        }
        __syncthreads();
        unsigned long long destroyed = 0;
        const bool many = nf >= 2 * NW;
        // a frontier vertex of count 0 lies in no clique of the current set:
        // nothing to enumerate (frontier counts do not change here), and at
        // level 0 that is every one of them; asking costs a load that a round of
        // few vertices would wait for (strips of 300 to 3,000 vertices, h = 2..4:
        // 9.1 ms, 10.5 when every round asks)
        if (k == 0) {
        } else if (B.h == 2) {
            for (uint32_t i = wid; i < nf; i += NW) {
                uint32_t v = F[i];
                if (many && B.deg[v] == 0) continue;
                for (uint32_t p = B.off[v] + lane; p < B.off[v + 1]; p += 32) {
                    uint32_t u = B.adj[p];
                    uint32_t s = B.st[u];
                    if (s == kAl) {
                        bdec(B, u, 1ull, k, G, &S.cnt2);
                        destroyed++;
                    } else if (s == kFr && u > v) {
                        destroyed++;
                    }
                }
            }
        } else {
            uint32_t* C = S.wbuf[wid];
            uint32_t* cnt = C + kBatchMaxDplus;
            // many frontier vertices: a warp each, those with long rows listed
            // for after; few, or listed: the block's warps share the neighbours of
            // one after another (a warp a vertex alone: 16 graphs G(600, 0.4),
            // h = 4, 665 ms against 536)
            const uint32_t* list = F;
            uint32_t nv = nf;
            for (bool each = many;; each = false) {
                for (uint32_t i = each ? wid : 0; i < nv; i += each ? NW : 1) {
                    const uint32_t v = list[i], b = B.off[v], e = B.off[v + 1];
                    if (each) {
                        if (B.deg[v] == 0) continue;
                        if (e - b > kBatchSharedRow) {
                            if (lane == 0) B.tmp[atomicAdd(&S.flag, 1u)] = v;
                            continue;
                        }
                    }
                    for (uint32_t p = b + (each ? 0 : wid); p < e; p += each ? 1 : NW) {
                        unsigned long long t = bitem<LPR>(B, v, B.adj[p], k, G, &S.cnt2, C, cnt);
                        if (lane == 0) destroyed += t;
                    }
                }
                if (!each) break;
                __syncthreads();
                list = B.tmp;
                nv = S.flag;
            }
        }
        destroyed = bsum<NT>(destroyed, S.red);
        for (uint32_t i = threadIdx.x; i < nf; i += NT) {
            uint32_t v = F[i];
            B.st[v] = kGo;
            B.core[v] = k;
            if (B.rnd) B.rnd[v] = r;
        }
        if (threadIdx.x == 0) S.mu_alive -= destroyed;
        __syncthreads();
        left -= nf;
        nf = S.cnt2;
        uint32_t* t = F;
        F = G;
        G = t;
        r++;
    }
    *nl = nlev;
    return k;
}

// a/b >= c/d in 128-bit arithmetic.
__device__ __forceinline__ bool bratio_ge(unsigned long long a, unsigned long long b,
                                          unsigned long long c, unsigned long long d) {
    unsigned long long lhi = __umul64hi(a, d), llo = a * d;
    unsigned long long rhi = __umul64hi(c, b), rlo = c * b;
    return lhi > rhi || (lhi == rhi && llo >= rlo);
}

// A warp's buffer for candidate sets of 33 .. kBatchWarpRows: ids, 64-bit
// counts, rows of row_stride(4) words, scratch of the node search.
constexpr uint32_t kBatchWarpRows = 128;
static_assert(3 * kBatchWarpRows + kBatchWarpRows * row_stride(4) + kWarpScratch <=
                  2 * kBatchMaxDplus + 64,
              "the warp's buffer holds the rows");
__device__ __forceinline__ unsigned long long* warp_counts64(uint32_t* buf) {
    return reinterpret_cast<unsigned long long*>(buf + kBatchWarpRows);
}

// Triangles of G[C], 32 < nc <= kBatchWarpRows, by one warp: the total; each
// candidate's count in warp_counts64(buf).  C is buf's start.
__device__ unsigned long long warp_triangles(const uint32_t* C, uint32_t nc, const uint32_t* off,
                                             const uint32_t* adj, const uint32_t* nb,
                                             uint32_t* buf) {
    const unsigned lane = lane_id();
    unsigned long long* c64 = warp_counts64(buf);
    uint32_t* rows = buf + 3 * kBatchWarpRows;
    const uint32_t W = (nc + 31) >> 5, Ws = row_stride(W);
    for (uint32_t i = lane; i < nc; i += 32) c64[i] = 0;
    for (uint32_t i = lane; i < nc * Ws; i += 32) rows[i] = 0;
    __syncwarp();
    const uint32_t cmax = C[nc - 1];
    for (uint32_t i = 0; i + 1 < nc; i++) {
        const uint32_t x = C[i];
        const uint32_t b = nb[x], e = off[x + 1];
        for (uint32_t p0 = b; p0 < e; p0 += 32) {
            const uint32_t p = p0 + lane;
            const uint32_t y = p < e ? adj[p] : kNone;
            if (y <= cmax) {
                const uint32_t pos = (uint32_t)lower_bound_u32(C, nc, y);
                if (pos < nc && C[pos] == y) {
                    atomicOr(&rows[i * Ws + (pos >> 5)], 1u << (pos & 31));
                    atomicOr(&rows[pos * Ws + (i >> 5)], 1u << (i & 31));
                }
            }
        }
    }
    __syncwarp();
    BitmapWarp B;
    B.rows = rows;
    B.W = W;
    B.Ws = Ws;
    B.cnt = c64;
    B.sP = rows + kBatchWarpRows * row_stride(4);
    B.list = reinterpret_cast<uint16_t*>(B.sP + kRowStrideMax);
    B.small = true;
    B.nd = nc;
    unsigned long long total = 0;
    for (uint32_t i = 0; i + 2 < nc; i++) {
        uint32_t P = B.row_word(i);
        const uint32_t iw = i >> 5;
        if (lane < iw) P = 0;
        else if (lane == iw) P &= (i & 31u) == 31u ? 0u : 0xffffffffu << ((i & 31u) + 1u);
        const unsigned long long c = warp_edges(B, P);
        if (c && lane == 0) B.credit(i, c);
        total += c;
    }
    __syncwarp();
    return total;
}

// ------------------------------------------------------------ the kernel
// LPR: lanes per row scan (the intersection tile; 32 / LPR rows at once per
// warp in the triangle listing and the h = 4 edge counts).
template <int NT, int LPR>
__global__ void __launch_bounds__(NT) k_batch(BatchArgs A) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    Smem<NT>& S = *reinterpret_cast<Smem<NT>*>(smem_raw);
    __shared__ uint32_t s_gi;
    const unsigned lane = lane_id(), wid = warp_id();
    Work W = carve(A.ws + (size_t)blockIdx.x * A.ws_stride, A.maxn, A.maxe);
    for (;;) {
        if (threadIdx.x == 0) s_gi = atomicAdd(A.queue, 1u);
        __syncthreads();
        uint32_t qi = s_gi;
        __syncthreads();
        if (qi >= A.count) break;
        const uint32_t gi = A.order[qi];
        const BatchDesc D = A.desc[gi];
        const uint32_t n = D.n;
        BatchRes R;
        memset(&R, 0, sizeof(R));
        if (n == 0 || n > kBatchMaxN || D.h < 2 || D.h > 4) {
            if (threadIdx.x == 0) {
                R.status = n == 0 ? kBOk : kBInvalid;
                A.res[gi] = R;
            }
            __syncthreads();
            continue;
        }
        // ---- CSR: endpoint counts, scatter, rows sorted, repeats dropped
        if (threadIdx.x == 0) S.flag = 0;
        for (uint32_t v = threadIdx.x; v < n; v += NT) W.fa[v] = 0;
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < D.m; e += NT) {
            const uint32_t u = A.src[D.e_off + e], v = A.dst[D.e_off + e];
            if (u >= n || v >= n) {
                S.flag = 1;
                continue;
            }
            if (u == v) continue;
            atomicAdd(&W.fa[u], 1u);
            atomicAdd(&W.fa[v], 1u);
        }
        __syncthreads();
        if (S.flag) {
            if (threadIdx.x == 0) {
                R.status = kBInvalid;
                A.res[gi] = R;
            }
            __syncthreads();
            continue;
        }
        (void)block_prefix<NT>(W.fa, n, W.roff, S);
        for (uint32_t v = threadIdx.x; v < n; v += NT) W.fa[v] = 0;
        __syncthreads();
        for (uint32_t e = threadIdx.x; e < D.m; e += NT) {
            const uint32_t u = A.src[D.e_off + e], v = A.dst[D.e_off + e];
            if (u == v) continue;
            W.k1[W.roff[u] + atomicAdd(&W.fa[u], 1u)] = v;
            W.k1[W.roff[v] + atomicAdd(&W.fa[v], 1u)] = u;
        }
        __syncthreads();
        block_sort_rows<NT>(W.k1, W.k2, W.roff, W.fa, n, W.fb, S);
        const uint32_t E = block_prefix<NT>(W.fa, n, W.off, S);
        for (uint32_t v = wid; v < n; v += NW) {
            const uint32_t from = W.roff[v], to = W.off[v], l = W.off[v + 1] - to;
            for (uint32_t j = lane; j < l; j += 32) W.adj[to + j] = W.k1[from + j];
        }
        __syncthreads();
        R.m_clean = E / 2;
        // ---- degeneracy peel (the h = 2 decomposition)
        for (uint32_t v = threadIdx.x; v < n; v += NT) W.deg[v] = W.off[v + 1] - W.off[v];
        __syncthreads();
        BPeel B2;
        B2.off = W.off;
        B2.adj = W.adj;
        B2.nplus = nullptr;
        B2.n = n;
        B2.h = 2;
        B2.deg = W.deg;
        B2.core = W.core;
        B2.rnd = W.rnd;
        B2.st = W.st;
        B2.alive = W.alive;
        B2.fa = W.fa;
        B2.fb = W.fb;
        B2.tmp = W.k2;
        B2.lk = W.lk;
        B2.lm = W.lm;
        B2.ls = W.ls;
        B2.mu0 = E / 2;
        uint32_t nl = 0;
        unsigned long long kmax = block_peel<NT, LPR>(B2, S, &nl);
        unsigned long long mu = E / 2;
        const unsigned long long* corev = W.core;   // caller ids
        if (D.h >= 3) {
            // ---- rank = (round, id), relabel, sorted rows
            for (uint32_t v = threadIdx.x; v < n; v += NT) W.k2[v] = (W.rnd[v] << 16) | v;
            __syncthreads();
            block_radix_sort<NT>(W.k2, W.k1, n, 32, S);
            for (uint32_t i = threadIdx.x; i < n; i += NT) {
                uint32_t o = W.k2[i] & 0xffffu;
                W.old_of[i] = o;
                W.new_of[o] = i;
            }
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < n; i += NT) {
                const uint32_t o = W.old_of[i];
                W.fa[i] = W.off[o + 1] - W.off[o];
            }
            __syncthreads();
            (void)block_prefix<NT>(W.fa, n, W.roff, S);
            for (uint32_t i = wid; i < n; i += NW) {
                const uint32_t from = W.off[W.old_of[i]], to = W.roff[i], l = W.roff[i + 1] - to;
                for (uint32_t j = lane; j < l; j += 32) W.radj[to + j] = W.new_of[W.adj[from + j]];
            }
            __syncthreads();
            block_sort_rows<NT>(W.radj, W.k1, W.roff, W.fa, n, W.fb, S);
            // N+(v): first entry above v; largest out-degree
            if (threadIdx.x == 0) S.cnt2 = 0;
            __syncthreads();
            for (uint32_t v = threadIdx.x; v < n; v += NT) {
                uint32_t b = W.roff[v], e = W.roff[v + 1];
                uint32_t s = b + (uint32_t)lower_bound_u32(W.radj + b, e - b, v + 1u);
                W.rsplit[v] = s;
                atomicMax(&S.cnt2, e - s);
            }
            __syncthreads();
            if (S.cnt2 > kBatchMaxDplus) {
                if (threadIdx.x == 0) {
                    R.status = kBUnsupported;
                    A.res[gi] = R;
                }
                __syncthreads();
                continue;
            }
            // ---- clique-degrees (warp per vertex, candidates in shared memory)
            for (uint32_t v = threadIdx.x; v < n; v += NT) W.deg[v] = 0;
            __syncthreads();
            unsigned long long mu_loc = 0;
            {
                uint32_t* C = S.wbuf[wid];
                uint32_t* cnt = C + kBatchMaxDplus;
                uint32_t* rows = cnt + kBatchMaxDplus;
                for (uint32_t u = wid; u < n; u += NW) {
                    uint32_t b = W.rsplit[u], e = W.roff[u + 1], d = e - b;
                    if (d < (uint32_t)(D.h - 1)) continue;
                    for (uint32_t i = lane; i < d; i += 32) {
                        C[i] = W.radj[b + i];
                        cnt[i] = 0;
                    }
                    __syncwarp();
                    unsigned long long tot = 0;
                    if (D.h == 3) {
                        // each hit of a row scan is a triangle {u, x, y}; the
                        // warp scans 32 / LPR rows at once
                        const unsigned gl = lane & (LPR - 1), gm = group_mask<LPR>();
                        unsigned long long mine = 0;
                        for (uint32_t i = lane / LPR; i < d; i += 32 / LPR) {
                            uint32_t x = C[i];
                            unsigned hits = 0;
                            for (uint32_t p = W.rsplit[x] + gl; p < W.roff[x + 1]; p += LPR) {
                                uint32_t y = W.radj[p];
                                uint32_t pos = (uint32_t)lower_bound_u32(C, d, y);
                                if (pos < d && C[pos] == y) { atomicAdd(&cnt[pos], 1u); hits++; }
                            }
                            hits = __reduce_add_sync(gm, hits);
                            if (gl == 0 && hits) atomicAdd(&cnt[i], hits);
                            if (gl == 0) mine += hits;
                        }
                        __syncwarp();
                        tot = warp_sum(mine);
                    } else if (d <= 32) {
                        // h = 4: triangles of G[C] by the one-word bitmap DFS
                        warp_rows32_ahead(C, d, W.roff + 1, W.radj, W.rsplit, rows);
                        tot = warp_dfs32(rows, d, 3, cnt);
                    } else if (d <= kBatchWarpRows) {
                        // h = 4, |C| <= 128: symmetric rows of at most four
                        // words and the edges of each upper row (cliques.cuh)
                        tot = warp_triangles(C, d, W.roff, W.radj, W.rsplit, S.wbuf[wid]);
                    } else {
                        // h = 4, larger |C|: every edge (x, y) of G[C] with x < y,
                        // and each common higher neighbour z of x and y in C
                        for (uint32_t i = 0; i < d; i++) {
                            uint32_t x = C[i];
                            const uint32_t* Nx = W.radj + W.rsplit[x];
                            uint32_t dx = W.roff[x + 1] - W.rsplit[x];
                            for (uint32_t p = 0; p < dx; p++) {
                                uint32_t y = Nx[p];
                                uint32_t py = (uint32_t)lower_bound_u32(C, d, y);
                                if (!(py < d && C[py] == y)) continue;
                                unsigned hits = 0;
                                for (uint32_t q = W.rsplit[y] + lane; q < W.roff[y + 1]; q += 32) {
                                    uint32_t z = W.radj[q];
                                    uint32_t pz = (uint32_t)lower_bound_u32(C, d, z);
                                    if (!(pz < d && C[pz] == z)) continue;
                                    uint32_t qx = (uint32_t)lower_bound_u32(Nx, dx, z);
                                    if (qx < dx && Nx[qx] == z) { atomicAdd(&cnt[pz], 1u); hits++; }
                                }
                                hits = __reduce_add_sync(0xffffffffu, hits);
                                if (lane == 0 && hits) {
                                    atomicAdd(&cnt[i], hits);
                                    atomicAdd(&cnt[py], hits);
                                }
                                tot += hits;
                            }
                        }
                    }
                    __syncwarp();
                    if (tot && D.h == 4 && d > 32 && d <= kBatchWarpRows) {
                        const unsigned long long* c64 = warp_counts64(S.wbuf[wid]);
                        for (uint32_t i = lane; i < d; i += 32)
                            if (c64[i]) atomicAdd(&W.deg[C[i]], c64[i]);
                    } else if (tot)
                        for (uint32_t i = lane; i < d; i += 32)
                            if (cnt[i]) atomicAdd(&W.deg[C[i]], (unsigned long long)cnt[i]);
                    if (lane == 0 && tot) {
                        atomicAdd(&W.deg[u], tot);
                        mu_loc += tot;
                    }
                    __syncwarp();
                }
            }
            mu = bsum<NT>(mu_loc, S.red);
            // ---- (k,Psi)-core peel on the ranked graph
            BPeel B;
            B.off = W.roff;
            B.adj = W.radj;
            B.nplus = W.rsplit;
            B.n = n;
            B.h = D.h;
            B.deg = W.deg;
            B.core = W.core;
            B.rnd = nullptr;
            B.st = W.st;
            B.alive = W.alive;
            B.fa = W.fa;
            B.fb = W.fb;
            B.tmp = W.k2;
            B.lk = W.lk;
            B.lm = W.lm;
            B.ls = W.ls;
            B.mu0 = mu;
            kmax = block_peel<NT, LPR>(B, S, &nl);
            // core numbers back to caller ids (k1 as 64-bit scratch is not
            // needed: write through old_of)
            for (uint32_t i = threadIdx.x; i < n; i += NT) W.deg[W.old_of[i]] = W.core[i];
            __syncthreads();
            corev = W.deg;
        }
        // ---- outputs: densest level (ties to larger k), k_max level
        {
            uint32_t best = 0xffffffffu;
            for (uint32_t j = threadIdx.x; j < nl; j += NT)
                if (best == 0xffffffffu || bratio_ge(W.lm[j], W.ls[j], W.lm[best], W.ls[best])) best = j;
            // block argmax with the same tie rule (larger index on ties)
            __shared__ uint32_t s_best[NT];
            s_best[threadIdx.x] = best;
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t bb = 0xffffffffu;
                for (int t = 0; t < NT; t++) {
                    uint32_t j = s_best[t];
                    if (j == 0xffffffffu) continue;
                    if (bb == 0xffffffffu) { bb = j; continue; }
                    bool ge = bratio_ge(W.lm[j], W.ls[j], W.lm[bb], W.ls[bb]);
                    bool le = bratio_ge(W.lm[bb], W.ls[bb], W.lm[j], W.ls[j]);
                    if ((ge && !le) || (ge && le && j > bb)) bb = j;
                }
                R.mu = mu;
                R.nlevels = nl;
                if (nl) {
                    R.kmax = W.lk[nl - 1];
                    R.kmax_core_size = W.ls[nl - 1];
                    R.kmax_core_mu = W.lm[nl - 1];
                    R.best_k = W.lk[bb];
                    R.densest_size = W.ls[bb];
                    R.densest_mu = W.lm[bb];
                }
                R.status = kBOk;
                A.res[gi] = R;
            }
            (void)kmax;
        }
        if (A.cores && D.core_off != ~0ull)
            for (uint32_t v = threadIdx.x; v < n; v += NT) A.cores[D.core_off + v] = corev[v];
        __syncthreads();
    }
}

}  // namespace
}  // namespace dsd

#include "batch_host.inc"
