// Level-synchronous (k,Psi)-core peeling with level statistics.
//
// Algorithm 3 removes one minimum clique-degree vertex at a time and lowers
// the clique-degree of every vertex sharing a clique instance with it, never
// below the removed vertex's value.  Here every alive vertex whose
// clique-degree is <= k leaves at once (the frontier F); each clique
// instance destroyed by F is credited once, to its smallest-id frontier
// member v, and lowers the count of each of its other members that are alive
// or frontier members (of larger id) by one.  A vertex whose count falls to
// <= k joins the next frontier at the same level; when no vertex is left at
// <= k, k jumps to the minimum alive count.  core(v) is the k at which v
// leaves.  A frontier member's count after its round is the number of
// cliques credited to it, so mu falls by the sum of those counts.  The first
// round of every level starts from the set R_k (Def. 6), whose size and
// clique count are recorded: these give the CoreApp outputs (the k_max core,
// Lemma 6) and the densest residual level (Pruning1, Sec. 5.1) without
// storing cliques.
//
// Levels are many and small (5,552 on the 1M-vertex Chung-Lu graph, h = 3;
// the last 8,000 vertices hold nearly all of them), and a round costs grid
// barriers and latency whatever its size, so taking the levels one after
// another is bound by their number.  R_t for any t is reached by one cascade
// from any R_s, s < t (remove everything below t, repeat), in a few rounds
// however many levels lie between.  So the peel has two phases:
//   1 -- bands.  The alive set is cut at a few thresholds t_1 < t_2 < ...,
//        chosen from a histogram of the counts at each jump; the vertices a
//        cascade removes form a band, a run of consecutive levels.  Each
//        vertex's count at its band's start is kept (c0).  A band of a
//        single level is finished here.
//   2 -- levels.  Every vertex of R_{t_i} \ R_{t_{i+1}} leaves between those
//        two sets, while R_{t_{i+1}} stays whole, so given c0 the bands do
//        not depend on one another: all of them are peeled level by level
//        side by side, a round of every band per grid round.  A clique
//        belongs to the lowest band among its members, and only members in
//        that band count it.
// The 1M-vertex graph, h = 3: 7,016 rounds one level at a time (86 ms), 587
// in the two phases (29 ms); R-MAT scale 17, h = 4: 8,232 and 428 (389 ms and
// 22 ms).  Bound by the latency of a round (barriers, row walks) and by the
// blocks that wait for the longest items of it.
//
// One persistent cooperative kernel runs every round; phases are separated
// by grid barriers whose waits are bounded in time (a wait that runs out
// records DSD_ERR_TIMEOUT and every block leaves).
//
// Phase 1, round r, F_r in global lists r mod 3:
//   P1  retire F_{r-1} (band); mark F_r as frontier                | barrier
//   J   (only if F_r is empty) compact the alive list, take the   |
//       minimum count and a histogram of the counts above k       | barrier
//       choose k; F_r = alive vertices with count <= k; when the   |
//       alive set has halved, drop removed vertices from the rows  |
//       of alive vertices                                         | barrier
//   P2  enumerate the cliques each v in F_r destroys; decrement   | barrier
//   P2b (h >= 4) candidate sets above warp_cand: warp groups and   |
//       blocks                                                    | barrier
//   or, h >= 3, a narrow frontier from a level's ninth round on:   |
//       block 0 runs rounds r, r + 1, ... alone (solo_rounds)     | barrier
// A cascade that grows too large or too long is undone (kBandMax,
// kBandRounds) and its first level taken alone.
// Phase 2, round r: each band has one owner block.
//   A   retire the band's frontier, find its next one (counts <= k, else
//       k = the least count: a new level), append it to F_r       | barrier
//   P2, P2b as above                                              | barrier
//
// Rows live in a private copy of the oriented CSR: row v is
// wadj[off[v] .. wend[v]).  In phase 1 N+(v) is its tail wadj[wnb[v] ..
// wend[v]); compaction rewrites a row in place (stable, so rows stay sorted)
// and moves wend/wnb.  For phase 2 every row keeps the entries of its own
// band and later ones, and N+(v) is read from the caller's rows (a
// compaction drops members of the bands peeled before it).
#include "bands.cuh"
#include "cliques.cuh"
#include "graph.cuh"
#include "xl.cuh"

#include <string.h>

namespace dsd {
namespace {

// state word: bits 0-1 the state, bit 2 kListedBit, bits 3-10 a bitmap slot
// (phase 1 only), bits 11-31 the band key (zero throughout phase 1)
enum : uint32_t { kAlive = 0, kFront = 1, kGone = 2 };
enum : uint32_t { kErrTimeout = 1, kErrBigOverflow = 2 };
constexpr uint32_t kSmallFront = 1024;
constexpr int kChunks = 4;              // 32-entry chunks of a row in flight per warp
constexpr uint32_t kWarpCand = 32;      // candidate sets a warp handles itself (h >= 4)
constexpr uint32_t kWarpWords = 3 * kWarpCand;   // a warp's candidates, counters, rows
// h = 4: a frontier vertex whose row holds at most kTinyRow entries goes to a
// warp, one of up to kBitmapMax to a block (or a few), which list the cliques
// of its whole neighbourhood at once; longer rows are taken one (vertex,
// neighbour) item at a time.
constexpr uint32_t kTinyRow = 32;
constexpr uint32_t kMaxSlices = 8;      // blocks sharing one such vertex
// Other h: the items of all frontier vertices are spread over the grid.  At h
// = 3 an item is one row walk (1M-vertex graph: 14 ms of phase 1 against 41 ms
// with a group of warps a vertex); at h = 5 the search inside an item has the
// short rows of a common neighbourhood (R-MAT scale 15: peel 22 ms against 28
// with whole rows).  In frontiers above kSmallFront only rows above kLongRow
// are spread, and those above kHubRow get bitmaps.
// h >= 3, phase 1: runs of rounds whose frontiers are at most kSoloFront
// vertices, all with rows of at most kSoloRow entries, go to block 0 alone
// (solo_rounds), at most kSoloRounds of them between two grid barriers, once a
// level or cascade has lasted kSoloAfter rounds: the last, narrow rounds of a
// power law's cascades (2-5 rounds) are as fast on the grid (cl50k, h = 3: 8.02
// ms; 8.12 with their narrow rounds in one block, 8.08 from the ninth on).
constexpr uint32_t kSoloFront = 64;
constexpr uint32_t kSoloRow = 16;
constexpr uint32_t kSoloRounds = 256;
constexpr uint32_t kSoloAfter = 8;
constexpr uint32_t kLongRow = 128;
constexpr uint32_t kHubRow = 512;
constexpr uint32_t kMidWords = 3 + kWarpCand;    // a mid item: v, w, |C|, C
constexpr int kGroupWarps = 8;                    // warps of a group taking one mid item
// h >= 4: a warp lists the cliques of a candidate set of at most this many
// vertices itself (default 4, dsd_set_peel_items); larger sets go to a warp
// group or a whole block after the next grid barrier.  Items are the round's
// critical path when one warp walks the rows of many candidates in turn: on
// R-MAT scale 21 the peel took 9.4 s (h = 4) and 20.5 s (h = 5) with the limit
// at 32, 5.2 s and 13.5 s at 4.
inline uint32_t warp_cand_limit(int h) {
    uint32_t w = peel_item_warp_limit();
    return h >= 4 ? (w < kWarpCand ? w : kWarpCand) : kWarpCand;
}
constexpr uint32_t kListedBit = 4;      // state word: frontier vertex on the row or heavy list
constexpr uint32_t kSlotShift = 3;      // state word: 1 + its neighbourhood bitmap slot
constexpr uint32_t kSlotMask = 0xffu;
constexpr uint32_t kKeyShift = 11;      // state word: band key

// Band keys: the j-th band of several levels has key 2j + 1, a vertex of a
// single-level band the key 2j with j the multi-level bands before it, so keys
// order the bands that phase 2 has to tell apart.
// h = 2: rounds taken one level at a time before the bands begin.  Levels are
// few there (at most the degeneracy), and a graph that is done in fewer rounds
// gains nothing: G(100,000, 0.0002) has 44 rounds in 7 levels (0.74 ms, 0.85
// with bands); the 50,000-vertex Chung-Lu graph 351 in 51 (3.85 -> 2.6 ms).
constexpr uint32_t kBandAfter2 = 64;
// h = 2: graphs of up to kOneBlockN vertices (12 bytes each fit shared memory)
// and kOneBlockAdj row entries go to one block (k_peel2_block).  Measured
// against the grid: G(2000, 0.005) 0.10 against 0.31 ms, power law with 10,000
// vertices 0.40 / 1.41, G(n, p) with 320,000 entries 0.47 / 0.53 and with
// 983,000 entries 1.05 / 0.61 ms.
constexpr uint32_t kOneBlockN = 16384;
constexpr uint64_t kOneBlockAdj = 400000;

__device__ __forceinline__ uint32_t st_of(uint32_t w) { return w & 3u; }

// Is x (state word wx) a member of the current set as seen from frontier
// vertex v of key kv, with frontier members of smaller id taken as gone?
// dec: x is also counting the cliques it shares with v (same band).
__device__ __forceinline__ bool cand_ok(uint32_t wx, uint32_t x, uint32_t kv, uint32_t v,
                                        bool& dec) {
    const uint32_t kx = wx >> kKeyShift, s = wx & 3u;
    dec = kx == kv && (s == kAlive || (s == kFront && x > v));
    return dec || kx > kv;
}

struct PeelCtrl {
    unsigned long long min_deg[2];
    uint32_t new_alive[2];
    uint32_t fcnt[3];
    uint32_t big_cnt[6];            // per round slot s: big items [s], mid items [3 + s]
    uint32_t hcnt[3];               // frontier vertices whose items are spread,
    uint32_t vcnt[3];               //   and whose rows are taken whole
    uint32_t vgrab[3];              // those (phase 2: frontier vertices) taken
    uint32_t grab[3];               // frontier vertices taken by warps
    uint32_t bgrab[6];              // big items [s] and mid items [3 + s] taken
    uint32_t hubcnt[2];             // bitmap slots asked for, by round parity
    uint32_t lrow[3];               // some frontier vertex has more than kSoloRow entries
    uint32_t solo[3];               // after solo_rounds: round, vertices retired, rounds of levels
    uint32_t busy[3];               // phase 2: bands with vertices left, by round
    unsigned long long destroyed;   // phase 1: cliques destroyed so far
    uint32_t pad0[4];
    uint32_t bar_count;
    uint32_t pad1[31];
    uint32_t bar_gen;
    uint32_t pad2[31];
    uint32_t error;
    uint32_t err_info;
    unsigned long long kmax;
    uint32_t nlevels;
    uint32_t rounds;                // rounds of the level-by-level peel
    unsigned long long items;
    unsigned long long bytes;       // algorithmic bytes (meter notes below)
    unsigned long long barrier_ns;  // block 0's time inside grid barriers
    uint32_t barriers;
    uint32_t compactions;
    uint32_t band_n;                // alive vertices when the bands began (0 = none)
    uint32_t band_round;            // round of phase 1 at that point
    uint32_t nbands;                // multi-level bands
    uint32_t grid_rounds;           // rounds executed, both phases
    unsigned long long phase2_ns;
    unsigned long long tph[8];      // block 0's time per phase (ns)
    uint32_t hist[2][kBins];        // counts above k at a jump, by jump parity
};

// Byte meter.  Every global-memory element the algorithm reads or writes is
// counted once per access: ids and state words 4 B, offsets 8 B, counters
// 8 B, an atomic read-modify-write 16 B, a binary search over a row of d
// entries floor(log2 d) + 1 probes of 4 B.  Shared-memory traffic is not
// counted, and bookkeeping that every block repeats counts once.
__device__ __forceinline__ unsigned probes(uint64_t d) {
    return d ? 64u - (unsigned)__clzll((long long)d) : 0u;
}

struct PeelParams {
    uint32_t n;
    int h;
    const uint64_t* off;   // row starts (read-only)
    uint32_t* wadj;        // private copy of the rows
    uint64_t* wend;        // row ends
    uint64_t* wnb;         // N+ starts (h >= 3)
    unsigned long long* deg;
    uint64_t* core;
    uint32_t* rnd;
    uint32_t* sl;          // state words
    uint32_t* alive[2];
    uint32_t* front[3];
    const uint32_t* nadj;  // the caller's rows (phase 2: N+(v) = nadj[nsplit[v] .. off[v + 1]))
    const uint64_t* nsplit;
    uint32_t* mem;         // vertices in the order phase 1 retired them
    uint32_t* band_of;     // band key
    unsigned long long* c0;  // count at the start of the band
    Band* bands;           // multi-level bands [kMaxBands]
    uint32_t* blkcnt;      // per-block counts of the final pass
    uint64_t* t_k;         // level records by position in mem (t_size 0: none)
    uint32_t* t_size;
    uint64_t* t_mu;
    uint32_t band_max;     // group levels into bands at <= this many alive (0 = never)
    uint2* big;
    uint64_t big_cap;
    uint32_t* heavy;       // phase 1, h >= 3: frontier vertices whose items are spread
    uint32_t* vlist;       //   (h = 4) or whose rows blocks take whole
    // Phase 1: frontier vertices with the longest rows get (up to hub_slots
    // per round) a bitmap of their neighbourhood over vertex ids, so that "x in N(v)" is one probe instead of a binary search.  Two
    // sets of hub_slots bitmaps of hub_words words, by round parity; hubs
    // lists the owners (2 x hub_slots).
    uint32_t* hub_bm;
    uint32_t* hubs;
    uint64_t hub_words;
    uint32_t hub_slots;    // 0 = no bitmaps
    uint64_t* lvl_k;
    uint32_t* lvl_size;
    uint64_t* lvl_mu;
    PeelCtrl* ctrl;
    uint64_t wait_ns;
    unsigned long long mu0;
    unsigned long long k0; // initial level: kstart - 1, or 0
    uint32_t cap;          // candidate sets are at most this (>= max |N+|, >= 32)
    uint32_t warp_cand;    // h >= 4: candidate sets a warp handles (<= kWarpCand); larger
                           // ones go to a warp group (mid items) or a block
    uint32_t gather_cap;   // a warp's candidate walk stops past this many
    uint32_t* mid;         // mid items: kMidWords words each (v, w, |C|, C)
    uint32_t mid_cap;      // 0: none (every set above warp_cand goes to a block)
    uint32_t* xl;          // per block (kMaxDepth + 1) * cap entries when cap > kBitmapMax
    int compact;           // drop removed vertices from rows as the graph shrinks
    uint64_t* snap;        // if set: each alive vertex's count at every level jump (the
                           // last one written is its count in its own (k,Psi)-core)
};

// ------------------------------------------------------------ barrier
__device__ bool grid_barrier(PeelCtrl* c, uint64_t wait_ns, unsigned long long& waited) {
    __shared__ uint32_t s_err;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t t_in = globaltimer_ns();
        volatile uint32_t* genp = &c->bar_gen;
        uint32_t gen = *genp;
        __threadfence();
        uint32_t arrived = atomicAdd(&c->bar_count, 1u) + 1u;
        if (arrived == gridDim.x) {
            c->bar_count = 0;
            __threadfence();
            atomicAdd(&c->bar_gen, 1u);
        } else {
            uint32_t spins = 0;
            while (*genp == gen) {
                if (((++spins) & 255u) == 0 && globaltimer_ns() - t_in > wait_ns) {
                    atomicOr(&c->error, kErrTimeout);
                    break;
                }
                if (*(volatile uint32_t*)&c->error) break;
            }
        }
        __threadfence();
        s_err = *(volatile uint32_t*)&c->error;
        waited += globaltimer_ns() - t_in;
    }
    __syncthreads();
    // one decision per block, so that its threads leave (or stay) together
    return s_err == 0;
}

// ------------------------------------------------------------ helpers

// N+ lists of the current phase: adj[nb[v] .. ne[v]).
struct NPlus {
    const uint32_t* adj;
    const uint64_t* nb;
    const uint64_t* ne;
};

// Lower the count of x, alive or frontier (state s), by c.  With a queue
// (phase 1) an alive vertex that falls to <= k joins the next frontier; phase
// 2 finds them by scanning the bands, and needs no old value.
__device__ __forceinline__ void lower(const PeelParams& P, uint32_t x, uint32_t s,
                                      unsigned long long c, unsigned long long k,
                                      uint32_t* next, uint32_t* next_cnt) {
    if (next && s == kAlive) {
        unsigned long long old = atomic_sub_u64(&P.deg[x], c);
        if (old > k && old - c <= k) {
            uint32_t at = atomicAdd(next_cnt, 1u);
            next[at] = x;
        }
    } else {
        atomic_sub_u64(&P.deg[x], c);
    }
}

// pre[0] = 0, pre[i+1] = sum of the current row lengths of F[0..i], for
// f <= kSmallFront entries (each thread owns kSmallFront/NT consecutive ones).
// ALL: every entry counts; else a frontier vertex marked gone (count 0) has
// no items.  Rows of at most `skip` entries count as empty.
template <int NT, bool ALL = false>
__device__ __forceinline__ void block_prefix_degrees(const PeelParams& P, const uint32_t* F,
                                                     uint32_t f, unsigned long long* pre,
                                                     unsigned long long* red, uint32_t skip = 0) {
    constexpr int E = kSmallFront / NT;
    unsigned long long d[E], sum = 0;
    uint32_t i0 = threadIdx.x * E;
#pragma unroll
    for (int q = 0; q < E; q++) {
        uint32_t i = i0 + q;
        d[q] = 0;
        if (i < f) {
            uint32_t v = F[i];
            if (ALL || st_of(P.sl[v]) == kFront) d[q] = P.wend[v] - P.off[v];
            if (d[q] <= skip) d[q] = 0;
        }
        sum += d[q];
    }
    unsigned lane = lane_id();
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane >= o) x += y;
    }
    if (lane == 31) red[warp_id()] = x;
    __syncthreads();
    unsigned long long before = 0;
    for (unsigned w = 0; w < warp_id(); w++) before += red[w];
    unsigned long long run = before + x - sum;
    if (threadIdx.x == 0) pre[0] = 0;
#pragma unroll
    for (int q = 0; q < E; q++) {
        run += d[q];
        if (i0 + q < f) pre[i0 + q + 1] = run;
    }
    __syncthreads();
}

// Candidates of frontier vertex v (key kv) among N+(w), in order (one warp):
// members of the current set (cand_ok) adjacent to v, tested on v's
// neighbourhood bitmap gbm over vertex ids when it has one, else by binary
// search in v's row.  kChunks chunks of the row are loaded at once.  MODE:
//   kGatherDirect (h = 3): each candidate closes the triangle {v, w, x}; a
//     counting candidate loses it on the spot; nothing is stored;
//   kGatherWarp: the first kWarpCand candidates go to C; the walk stops as
//     soon as there are more than P.gather_cap (the item then needs a block).
// Returns the number of candidates seen; anyd: some of this lane's count.
enum { kGatherDirect = 0, kGatherWarp = 1 };

template <int MODE>
__device__ __forceinline__ void take_candidate(const PeelParams& P, bool ok, bool dec, uint32_t s,
                                               uint32_t x, uint32_t* C, uint32_t& nc, bool& anyd,
                                               unsigned long long k, uint32_t* next,
                                               uint32_t* next_cnt, unsigned long long& bytes) {
    unsigned lane = lane_id();
    unsigned bal = __ballot_sync(0xffffffffu, ok);
    if (ok && dec) anyd = true;
    if (MODE == kGatherDirect) {
        if (ok && dec) {
            lower(P, x, s, 1ull, k, next, next_cnt);
            bytes += 16;
        }
    } else {
        uint32_t at = nc + __popc(bal & ((1u << lane) - 1u));
        if (ok && at < kWarpCand) C[at] = x;
    }
    nc += __popc(bal);
}

template <int MODE>
__device__ __forceinline__ uint32_t gather_candidates(const PeelParams& P, const NPlus& R,
                                                      uint32_t v, uint32_t kv, uint32_t w,
                                                      uint32_t* C, const uint32_t* gbm,
                                                      bool& anyd, unsigned long long k,
                                                      uint32_t* next, uint32_t* next_cnt,
                                                      unsigned long long& bytes) {
    unsigned lane = lane_id();
    const uint32_t* Nv = P.wadj + P.off[v];
    uint64_t dv = P.wend[v] - P.off[v];
    uint64_t b = R.nb[w], e = R.ne[w];
    const uint64_t dw = e - b;
    const unsigned pr = probes(dv);
    uint32_t nc = 0;
    // Walk the shorter side: the entries of N(v) above w, each searched in
    // N+(w), when that costs fewer probes than walking N+(w).
    const uint64_t cost_w = gbm ? dw : dw * pr;
    const bool own = dv * probes(dw) < cost_w;
    const uint32_t* L = own ? Nv : R.adj + b;       // the list walked
    const uint64_t len = own ? dv : dw;
    const uint32_t* S = own ? R.adj + b : Nv;       // the list searched
    const uint64_t slen = own ? dw : dv;
    const unsigned ps = probes(slen);
    const uint32_t* bm = own ? nullptr : gbm;
    for (uint64_t p0 = own ? lower_bound_u32(Nv, dv, w + 1u) : 0; p0 < len; p0 += 32 * kChunks) {
        uint32_t xs[kChunks], ws[kChunks];
#pragma unroll
        for (int u = 0; u < kChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            xs[u] = p < len ? L[p] : 0u;
        }
#pragma unroll
        for (int u = 0; u < kChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            ws[u] = p < len ? P.sl[xs[u]] : (uint32_t)kGone;
        }
#pragma unroll
        for (int u = 0; u < kChunks; u++) {
            uint64_t p = p0 + u * 32 + lane;
            bool ok = false, dec = false;
            uint32_t x = xs[u];
            if (p < len) {
                bytes += 8;
                if (cand_ok(ws[u], x, kv, v, dec)) {
                    if (bm) {
                        ok = (bm[x >> 5] >> (x & 31)) & 1u;
                        bytes += 4;
                    } else {
                        uint64_t pos = lower_bound_u32(S, slen, x);
                        ok = pos < slen && S[pos] == x;
                        bytes += 4ull * ps;
                    }
                }
            }
            take_candidate<MODE>(P, ok, dec, st_of(ws[u]), x, C, nc, anyd, k, next, next_cnt,
                                 bytes);
        }
        if (MODE == kGatherWarp && nc > P.gather_cap) return nc;
    }
    return nc;
}

// One (v, w) work item of a frontier vertex v with h >= 3: the cliques
// {v, w, ...} whose members other than v are candidates of v (in the current
// set, N+(.) from R) and whose smallest such member is w.  Executed by one warp; C, cnt, rows are the
// warp's kWarpCand-entry buffers.  Candidate sets above P.warp_cand (h >= 4)
// are queued, as mid items with their candidates when at most kWarpCand
// (`big_cnt + 3` counts them), else as big items for a block.
template <int HC>
__device__ void process_vw(const PeelParams& P, const NPlus& R, uint32_t v, uint32_t w,
                           unsigned long long k, uint32_t* next, uint32_t* next_cnt, uint32_t* C,
                           unsigned* cnt, uint32_t* rows, uint32_t* big_cnt, const uint32_t* gbm,
                           unsigned long long& bytes) {
    unsigned lane = lane_id();
    const uint32_t kv = P.sl[v] >> kKeyShift, ww = P.sl[w];
    bool dec_w;
    if (lane == 0) bytes += 4 + 4;   // w, its state word
    if (!cand_ok(ww, w, kv, v, dec_w)) return;
    if (lane == 0) bytes += 16;      // the bounds of N+(w)
    const int r = HC == 3 ? 1 : P.h - 2;
    unsigned long long tot = 0;
    bool anyd = false;
    if (r == 1) {
        tot = gather_candidates<kGatherDirect>(P, R, v, kv, w, C, gbm, anyd, k, next, next_cnt,
                                               bytes);
    } else {
        uint32_t nc = gather_candidates<kGatherWarp>(P, R, v, kv, w, C, gbm, anyd, k, next,
                                                     next_cnt, bytes);
        __syncwarp();
        if (nc < (uint32_t)r) return;
        // none count -- known only of a complete walk: one that stopped past
        // gather_cap has not seen the rest (a block looks again, process_big)
        if (nc <= P.gather_cap && !dec_w && !__any_sync(0xffffffffu, anyd)) return;
        if (nc > P.warp_cand) {
            // mid item: its candidates go with it to a warp group; else a block
            if (nc <= kWarpCand && P.mid_cap) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(big_cnt + 3, 1u);
                at = __shfl_sync(0xffffffffu, at, 0);
                if (at < P.mid_cap) {
                    uint32_t* rec = P.mid + (size_t)at * kMidWords;
                    if (lane < nc) rec[3 + lane] = C[lane];
                    if (lane == 0) {
                        rec[0] = v;
                        rec[1] = w;
                        rec[2] = nc;
                        bytes += 12 + 4ull * nc;
                    }
                    return;
                }
            }
            if (lane == 0) {
                uint32_t at = atomicAdd(big_cnt, 1u);
                if (at < P.big_cap) P.big[at] = make_uint2(v, w);
                else atomicOr(&P.ctrl->error, kErrBigOverflow);
            }
            return;
        }
        for (uint32_t i = lane; i < nc; i += 32) cnt[i] = 0;
        __syncwarp();
        if (r == 2) {
            // edges of G[C]: each is a clique {v, w, x, y}
            const uint32_t cmax = C[nc - 1];
            for (uint32_t i = 0; i + 1 < nc; i++) {
                uint32_t x = C[i];
                uint64_t xb = R.nb[x], xe = R.ne[x], xr = xe;
                unsigned hits = scan_row_hits(C, nc, cmax, R.adj, xb, xe, cnt, &xr);
                if (lane == 0) bytes += 16 + 4ull * (xr - xb);
                hits = __reduce_add_sync(0xffffffffu, hits);
                if (lane == 0 && hits) atomicAdd(&cnt[i], hits);
                tot += hits;
            }
        } else {
            if (lane == 0)
                for (uint32_t i = 0; i < nc; i++)
                    bytes += 16 + 4ull * (R.ne[C[i]] - R.nb[C[i]]);
            warp_build_rows32(C, nc, R.ne, R.adj, R.nb, rows);
            tot = warp_dfs32(rows, nc, r, cnt);
        }
        __syncwarp();
        if (tot)
            for (uint32_t i = lane; i < nc; i += 32) {
                uint32_t x = C[i];
                if (cnt[i]) {
                    bool dec;
                    const uint32_t wx = P.sl[x];
                    bytes += 4;
                    (void)cand_ok(wx, x, kv, v, dec);
                    if (dec) {
                        lower(P, x, st_of(wx), (unsigned long long)cnt[i], k, next, next_cnt);
                        bytes += 16;
                    }
                }
            }
        __syncwarp();
    }
    if (tot && lane == 0 && dec_w) {
        lower(P, w, st_of(ww), tot, k, next, next_cnt);
        bytes += 16;
    }
}

// h = 3, phase 2: one pair (v, u) of a frontier vertex v and a counting
// neighbour u of the same band (state word wu): u loses the triangles {v, u,
// x} with x in the current set.  Rows hold no member of an earlier band, so
// the members of a later band are never enumerated on their own account:
// only pairs inside a band cost anything.  One warp; the shorter of the two
// rows is read and searched for in the longer.
__device__ __forceinline__ void process_pair(const PeelParams& P, uint32_t v, uint32_t kv,
                                             uint32_t u, unsigned long long& bytes) {
    const unsigned lane = lane_id();
    const uint32_t* A = P.wadj + P.off[v];
    uint64_t da = P.wend[v] - P.off[v];
    const uint32_t* B = P.wadj + P.off[u];
    uint64_t db = P.wend[u] - P.off[u];
    if (db < da) {
        const uint32_t* t = A;
        A = B;
        B = t;
        const uint64_t td = da;
        da = db;
        db = td;
    }
    const unsigned pr = probes(db);
    unsigned hits = 0;
    for (uint64_t p0 = 0; p0 < da; p0 += 32 * kChunks) {
        uint32_t xs[kChunks], ws[kChunks];
#pragma unroll
        for (int q = 0; q < kChunks; q++) {
            uint64_t p = p0 + q * 32 + lane;
            xs[q] = p < da ? A[p] : 0u;
        }
#pragma unroll
        for (int q = 0; q < kChunks; q++) {
            uint64_t p = p0 + q * 32 + lane;
            ws[q] = p < da ? P.sl[xs[q]] : (uint32_t)kGone;
        }
#pragma unroll
        for (int q = 0; q < kChunks; q++) {
            uint64_t p = p0 + q * 32 + lane;
            bool dec;
            if (p < da) {
                bytes += 8;
                if (cand_ok(ws[q], xs[q], kv, v, dec)) {
                    uint64_t pos = lower_bound_u32(B, db, xs[q]);
                    hits += pos < db && B[pos] == xs[q];
                    bytes += 4ull * pr;
                }
            }
        }
    }
    hits = __reduce_add_sync(0xffffffffu, hits);
    if (lane == 0 && hits) {
        atomic_sub_u64(&P.deg[u], (unsigned long long)hits);
        bytes += 16 + 16;
    }
}

// A (v, w) item whose candidate set exceeds 32 vertices (h >= 4): one block,
// bitmap rows of G[C] and a warp-level DFS per starting candidate.  When
// N+(w) holds more than kBitmapMax entries (degeneracy above 1024) the
// candidates are gathered into the block's global scratch; a set that still
// exceeds kBitmapMax is split by its next member (xl.cuh).
__device__ void process_big(const PeelParams& P, const NPlus& R, uint32_t v, uint32_t w,
                            unsigned long long k, uint32_t* next, uint32_t* next_cnt,
                            uint32_t* smem, const uint32_t* gbm, unsigned long long& bytes) {
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(smem);
    uint32_t* C = smem + 2 * kBitmapMax;
    uint32_t* rows = smem + bitmap_rows_at(kBitmapMax);
    uint32_t* scratch = smem + bitmap_scratch_at(kBitmapMax);
    __shared__ uint32_t s_nc;
    __shared__ uint32_t s_next;
    __shared__ unsigned long long s_tot;
    __shared__ uint32_t s_flag[kBitmapMax / 32], s_at[kBitmapMax / 32];
    __shared__ uint32_t s_w[32], s_t2;
    const unsigned lane = lane_id(), nw = blockDim.x >> 5;
    const uint32_t kv = P.sl[v] >> kKeyShift, ww = P.sl[w];
    bool dec_w;
    (void)cand_ok(ww, w, kv, v, dec_w);
    const uint64_t b = R.nb[w], e = R.ne[w];
    const uint32_t* Nv = P.wadj + P.off[v];
    const uint64_t dv = P.wend[v] - P.off[v];
    const unsigned pr = probes(dv);
    if (e - b > kBitmapMax) {
        // oversized N+(w): gather in order into the block's global scratch
        uint32_t* G0 = P.xl + (size_t)blockIdx.x * (kMaxDepth + 1) * P.cap;
        const uint32_t nc = block_filter(
            R.adj + b, e - b, G0,
            [&](uint32_t x) {
                bool dec;
                if (!cand_ok(P.sl[x], x, kv, v, dec)) return false;
                if (gbm) return ((gbm[x >> 5] >> (x & 31)) & 1u) != 0u;
                uint64_t pos = lower_bound_u32(Nv, dv, x);
                return pos < dv && Nv[pos] == x;
            },
            s_w, &s_t2);
        if (threadIdx.x == 0) bytes += (8ull + 4ull * pr) * (e - b) + 24;
        if (nc > kBitmapMax) {
            if (threadIdx.x == 0) s_tot = 0;
            __syncthreads();
            xl_cliques(
                G0, nc, P.h - 2, R.nb, R.ne, R.adj, G0 + P.cap, P.cap, smem,
                [&](uint32_t x, unsigned long long c) {
                    bool dec;
                    const uint32_t wx = P.sl[x];
                    (void)cand_ok(wx, x, kv, v, dec);
                    if (dec) lower(P, x, st_of(wx), c, k, next, next_cnt);
                },
                [&](unsigned long long c) { s_tot += c; });
            __syncthreads();
            if (threadIdx.x == 0 && s_tot && dec_w)
                lower(P, w, st_of(ww), s_tot, k, next, next_cnt);
            __syncthreads();
            return;
        }
        for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) C[i] = G0[i];
        if (threadIdx.x == 0) {
            s_nc = nc;
            s_next = 0;
            s_tot = 0;
        }
        __syncthreads();
        if (nc < (uint32_t)(P.h - 2)) return;
        goto bitmap;
    }
    {
    // candidates of v among N+(w), all warps at once: warp c tests the c-th
    // run of 32 entries, the runs' hit masks are compacted in order
    const uint32_t runs = (uint32_t)((e - b + 31) >> 5);   // <= kBitmapMax / 32
    for (uint32_t c = warp_id(); c < runs; c += nw) {
        const uint64_t p = b + (uint64_t)c * 32 + lane;
        bool ok = false;
        if (p < e) {
            const uint32_t x = R.adj[p];
            bool dec;
            bytes += 8;
            if (cand_ok(P.sl[x], x, kv, v, dec)) {
                if (gbm) {
                    ok = (gbm[x >> 5] >> (x & 31)) & 1u;
                    bytes += 4;
                } else {
                    uint64_t pos = lower_bound_u32(Nv, dv, x);
                    ok = pos < dv && Nv[pos] == x;
                    bytes += 4ull * pr;
                }
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) s_flag[c] = bal;
    }
    __syncthreads();
    if (warp_id() == 0) {
        uint32_t tot = 0;
        for (uint32_t c0 = 0; c0 < runs; c0 += 32) {
            const uint32_t c = c0 + lane;
            uint32_t x = c < runs ? (uint32_t)__popc(s_flag[c]) : 0u, inc = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
                if ((int)lane >= o) inc += y;
            }
            if (c < runs) s_at[c] = tot + inc - x;
            tot += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) {
            s_nc = tot;
            s_next = 0;
            s_tot = 0;
            bytes += 4 + 4 + 16;
        }
    }
    __syncthreads();
    for (uint32_t c = warp_id(); c < runs; c += nw) {
        const unsigned bal = s_flag[c];
        if ((bal >> lane) & 1u)
            C[s_at[c] + __popc(bal & ((1u << lane) - 1u))] = R.adj[b + (uint64_t)c * 32 + lane];
    }
    __syncthreads();
    }
bitmap:
    uint32_t nc = s_nc;
    uint32_t W = (nc + 31) >> 5;
    {
        // nothing to do unless w or some candidate counts these cliques
        bool any = dec_w;
        for (uint32_t i = threadIdx.x; i < nc && !any; i += blockDim.x)
            (void)cand_ok(P.sl[C[i]], C[i], kv, v, any);
        if (!__syncthreads_or(any)) return;
    }
    for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
        cnt[i] = 0;
        bytes += 16 + 4ull * (R.ne[C[i]] - R.nb[C[i]]);
    }
    for (uint32_t i = threadIdx.x; i < nc * row_stride(W); i += blockDim.x) rows[i] = 0;
    __syncthreads();
    block_window(C, nc, scratch - kWindowWords);
    __syncthreads();
    block_build_rows(C, nc, W, R.ne, R.adj, R.nb, rows, scratch - kWindowWords);
    __syncthreads();
    unsigned long long mine = block_dfs(rows, nc, W, P.h - 2, cnt, &s_next, scratch);
    if (mine) atomicAdd(&s_tot, mine);
    __syncthreads();
    unsigned long long tot = s_tot;
    if (tot) {
        for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
            uint32_t x = C[i];
            if (!cnt[i]) continue;
            bool dec;
            const uint32_t wx = P.sl[x];
            (void)cand_ok(wx, x, kv, v, dec);
            if (dec) {
                lower(P, x, st_of(wx), cnt[i], k, next, next_cnt);
                bytes += 20;
            }
        }
        if (threadIdx.x == 0 && dec_w) lower(P, w, st_of(ww), tot, k, next, next_cnt);
    }
    __syncthreads();
}

__device__ __forceinline__ void group_bar(uint32_t id, uint32_t threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Mid items (h >= 4; candidate sets of warp_cand + 1 .. 32 vertices, listed
// by the warp that found them): groups of kGroupWarps warps take them from
// *grab, several per block at once.  The group's warps build the one-word
// rows of G[C] side by side (one candidate's list each), its first warp
// lists the cliques of G[C] (warp_dfs32), and the alive members are lowered.
// Group g synchronises on named barrier 1 + g.
template <int NT>
__device__ void drain_mid(const PeelParams& P, const NPlus& R, uint32_t nm, uint32_t* grab,
                          unsigned long long k, uint32_t* next, uint32_t* next_cnt,
                          unsigned long long& bytes) {
    constexpr int NG = NT / 32 / kGroupWarps;
    struct MidBuf {
        uint32_t C[kWarpCand];
        unsigned cnt[kWarpCand];
        uint32_t rows[kWarpCand];
        uint32_t i;
        unsigned long long tot;
    };
    __shared__ MidBuf s_mb[NG];
    const unsigned lane = lane_id(), wid = warp_id();
    const uint32_t grp = wid / kGroupWarps, gw = wid % kGroupWarps;
    const uint32_t bar = 1u + grp, nth = kGroupWarps * 32u;
    MidBuf& B = s_mb[grp];
    const int r = P.h - 2;
    for (;;) {
        if (gw == 0 && lane == 0) B.i = atomicAdd(grab, 1u);
        group_bar(bar, nth);
        const uint32_t i = B.i;
        if (i >= nm) break;
        const uint32_t* rec = P.mid + (size_t)i * kMidWords;
        const uint32_t v = rec[0], w = rec[1], nc = rec[2];
        const uint32_t kv = P.sl[v] >> kKeyShift;
        if (gw == 0) {
            B.C[lane] = lane < nc ? rec[3 + lane] : 0u;
            B.cnt[lane] = 0;
            B.rows[lane] = 0;
        }
        group_bar(bar, nth);
        const uint32_t cmax = B.C[nc - 1];
        for (uint32_t x = gw; x + 1 < nc; x += kGroupWarps) {
            const uint32_t y = B.C[x];
            const uint32_t bits = warp_row32(B.C, nc, cmax, y, R.adj, R.nb[y], R.ne[y]);
            if (lane == 0) {
                B.rows[x] = bits;
                bytes += 16 + 4ull * (R.ne[y] - R.nb[y]);
            }
        }
        group_bar(bar, nth);
        if (gw == 0) {
            const unsigned long long t = warp_dfs32(B.rows, nc, r, B.cnt);
            if (lane == 0) B.tot = t;
        }
        group_bar(bar, nth);
        const unsigned long long tot = B.tot;
        if (tot) {
            const uint32_t t = gw * 32 + lane;
            if (t < nc && B.cnt[t]) {
                const uint32_t x = B.C[t];
                const uint32_t wx = P.sl[x];
                bool dec;
                (void)cand_ok(wx, x, kv, v, dec);
                if (dec) {
                    lower(P, x, st_of(wx), (unsigned long long)B.cnt[t], k, next, next_cnt);
                    bytes += 20;
                }
            }
            if (gw == 0 && lane == 0) {
                const uint32_t ww = P.sl[w];
                bool dec;
                (void)cand_ok(ww, w, kv, v, dec);
                if (dec) lower(P, w, st_of(ww), tot, k, next, next_cnt);
            }
        }
        group_bar(bar, nth);   // B is rewritten by the next item
    }
}

// Drop removed vertices (phase 2, where every key is set: members of earlier
// bands) from row v in place (one warp); rows stay sorted.
__device__ __forceinline__ void compact_row(const PeelParams& P, uint32_t v, uint32_t kv,
                                            unsigned long long& bytes) {
    unsigned lane = lane_id();
    uint64_t b = P.off[v], e = P.wend[v];
    uint64_t outp = b;
    uint64_t below = 0;   // kept entries smaller than v
    for (uint64_t p0 = b; p0 < e; p0 += 32) {
        uint64_t p = p0 + lane;
        uint32_t x = 0;
        bool keep = false;
        if (p < e) {
            x = P.wadj[p];
            const uint32_t wx = P.sl[x], kx = wx >> kKeyShift;
            keep = kx > kv || (kx == kv && st_of(wx) != kGone);
        }
        unsigned bal = __ballot_sync(0xffffffffu, keep);
        unsigned lt = __ballot_sync(0xffffffffu, keep && x < v);
        // every lane has read its entry before any lane writes
        if (keep) P.wadj[outp + __popc(bal & ((1u << lane) - 1u))] = x;
        outp += __popc(bal);
        below += __popc(lt);
        __syncwarp();
    }
    bytes += 8ull * (e - b) + 4ull * (outp - b);
    if (lane == 0) {
        P.wend[v] = outp;
        P.wnb[v] = b + below;
        bytes += 16;
    }
}

// Phase 1: the neighbourhood bitmap of frontier vertex v for rounds of
// parity par, or null if v has none.
__device__ __forceinline__ const uint32_t* hub_bm_of(const PeelParams& P, uint32_t v,
                                                    uint32_t par) {
    if (!P.hub_slots) return nullptr;
    uint32_t slot = (P.sl[v] >> kSlotShift) & kSlotMask;
    return slot ? P.hub_bm + ((size_t)par * P.hub_slots + (slot - 1)) * P.hub_words : nullptr;
}

// Phase 1, marking v as a member of frontier F_r: its state word (gone at
// once if it lies in no clique of the current set: nothing is enumerated
// from it).  h >= 3: cls = 1 for rows that blocks take whole, 2 for rows whose
// items are spread, both kListedBit; the longest of the latter get, while
// slots of this parity last, 1 + a bitmap slot (the owner goes to the
// parity's hub list).
template <int HC>
__device__ __forceinline__ uint32_t front_word(const PeelParams& P, PeelCtrl* c, uint32_t v,
                                               uint32_t par, uint32_t& cls, bool& lrow) {
    cls = 0;
    lrow = false;
    if (P.deg[v] == 0) return kGone;
    if (HC == 2) return kFront;
    const uint64_t d = P.wend[v] - P.off[v];
    lrow = d > kSoloRow;
    if (HC != 4) cls = d > kLongRow ? 2u : 0u;
    else cls = d > kBitmapMax ? 2u : (d > kTinyRow ? 1u : 0u);
    uint32_t w = kFront | (cls ? kListedBit : 0u);
    if (P.hub_slots && d > (HC == 4 ? kBitmapMax : kHubRow)) {
        uint32_t at = atomicAdd(&c->hubcnt[par], 1u);
        if (at < P.hub_slots) {
            P.hubs[par * P.hub_slots + at] = v;
            w |= (at + 1u) << kSlotShift;
        }
    }
    return w;
}

// Sets (or, clear = true, zeroes the words of) the bitmaps of the hubs of
// parity par over their rows; the rows' entries are flattened over every
// thread of the grid.  Every thread of every block calls it.
template <int NT>
__device__ __forceinline__ void hub_bitmaps(const PeelParams& P, uint32_t nhub, uint32_t par,
                                            bool clear, unsigned long long* s_pre,
                                            unsigned long long* s_red,
                                            unsigned long long& bytes) {
    const uint32_t* H = P.hubs + (size_t)par * P.hub_slots;
    block_prefix_degrees<NT, true>(P, H, nhub, s_pre, s_red);
    const unsigned long long T = s_pre[nhub];
    const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t gthreads = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = gtid; t < T; t += gthreads) {
        uint32_t lo = 0, hi = nhub;
        while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (s_pre[mid] <= t) lo = mid; else hi = mid;
        }
        uint32_t v = H[lo];
        uint32_t x = P.wadj[P.off[v] + (t - s_pre[lo])];
        uint32_t* bm = P.hub_bm + ((size_t)par * P.hub_slots + lo) * P.hub_words;
        if (clear) bm[x >> 5] = 0u;   // every set bit belongs to a row entry
        else atomicOr(&bm[x >> 5], 1u << (x & 31));
        bytes += 4 + 16;
    }
    __syncthreads();   // s_pre is reused afterwards
}

// Every clique through frontier vertex v of a short row (at most kTinyRow
// entries), by one warp: the members of the current set among its neighbours
// and the (h-1)-cliques they span; C, cnt, rows are the warp's buffers.
template <int HC, bool AHEAD = false>
__device__ void process_tiny(const PeelParams& P, const NPlus& R, uint32_t v,
                             unsigned long long k, uint32_t* next, uint32_t* next_cnt,
                             uint32_t* C, unsigned* cnt, uint32_t* rows,
                             unsigned long long& bytes) {
    const unsigned lane = lane_id();
    const uint32_t kv = P.sl[v] >> kKeyShift;
    const uint64_t b = P.off[v];
    const uint32_t len = (uint32_t)(P.wend[v] - b);
    const int r = HC == 3 ? 2 : P.h - 1;
    uint32_t x = 0, wx = 0;
    bool ok = false, dec = false;
    if (lane < len) {
        x = P.wadj[b + lane];
        wx = P.sl[x];
        ok = cand_ok(wx, x, kv, v, dec);
        bytes += 8;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, ok);
    const uint32_t nc = __popc(bal), at = __popc(bal & ((1u << lane) - 1u));
    if (nc < (uint32_t)r || !__any_sync(0xffffffffu, ok && dec)) return;
    if (ok) C[at] = x;
    cnt[lane] = 0;
    __syncwarp();
    if (lane < nc) bytes += 16 + 4ull * (R.ne[C[lane]] - R.nb[C[lane]]);
    if (AHEAD) {
        // nothing else hides the latency of a round of few vertices
        warp_rows32_ahead(C, nc, R.ne, R.adj, R.nb, rows);
        (void)warp_dfs32(rows, nc, r, cnt);
    } else if (r == 2) {
        const uint32_t cmax = C[nc - 1];
        for (uint32_t i = 0; i + 1 < nc; i++) {
            const uint32_t y = C[i];
            unsigned hits = scan_row_hits(C, nc, cmax, R.adj, R.nb[y], R.ne[y], cnt);
            hits = __reduce_add_sync(0xffffffffu, hits);
            if (lane == 0 && hits) atomicAdd(&cnt[i], hits);
        }
    } else {
        warp_build_rows32(C, nc, R.ne, R.adj, R.nb, rows);
        (void)warp_dfs32(rows, nc, r, cnt);
    }
    __syncwarp();
    if (ok && dec && cnt[at]) {
        lower(P, x, st_of(wx), (unsigned long long)cnt[at], k, next, next_cnt);
        bytes += 16;
    }
    __syncwarp();
}

// h = 4: the cliques through frontier vertex v (a row of at most kBitmapMax
// entries), by a block: bitmap rows of its whole neighbourhood once, instead
// of once for each (v, w) item, then the (h-1)-cliques in it.  Rows are
// numbered with the nd neighbours that count these cliques first (phase 2:
// those of v's band), and only they are first members, so that a clique whose
// other members all lie in later bands is never listed.  Slice s of S: the
// first members s, s + S, ... (several blocks share one vertex when there are
// few).  smem: bitmap_words(kBitmapMax, warps) words and kBitmapMax 16-bit
// row numbers.  R-MAT scale 17: peel 93 -> 22 ms.
__device__ void process_row(const PeelParams& P, const NPlus& R, uint32_t v, uint32_t s,
                            uint32_t S, unsigned long long k, uint32_t* next, uint32_t* next_cnt,
                            uint32_t* smem, unsigned long long& bytes) {
    __shared__ uint32_t s_flag[kBitmapMax / 32], s_dec[kBitmapMax / 32];
    __shared__ uint32_t s_next;
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(smem);
    uint32_t* C = smem + 2 * kBitmapMax;
    uint32_t* rows = smem + bitmap_rows_at(kBitmapMax);
    uint32_t* scratch = smem + bitmap_scratch_at(kBitmapMax);
    const unsigned lane = lane_id(), nw = blockDim.x >> 5;
    const uint32_t kv = P.sl[v] >> kKeyShift;
    const uint64_t b = P.off[v];
    const uint32_t len = (uint32_t)(P.wend[v] - b), runs = (len + 31) >> 5;
    const int r = P.h - 1;
    for (uint32_t c = warp_id(); c < runs; c += nw) {
        const uint32_t p = c * 32 + lane;
        bool ok = false, dec = false;
        if (p < len) {
            const uint32_t x = P.wadj[b + p];
            ok = cand_ok(P.sl[x], x, kv, v, dec);
            bytes += 8;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        const unsigned bad = __ballot_sync(0xffffffffu, ok && dec);
        if (lane == 0) {
            s_flag[c] = bal;
            s_dec[c] = bad;
        }
    }
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    const uint32_t f = lane < runs ? s_flag[lane] : 0u, g = lane < runs ? s_dec[lane] : 0u;
    uint32_t inc = __popc(f), dinc = __popc(g);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        uint32_t z = __shfl_up_sync(0xffffffffu, dinc, o);
        if ((int)lane >= o) {
            inc += y;
            dinc += z;
        }
    }
    const uint32_t ex = inc - __popc(f), nc = __shfl_sync(0xffffffffu, inc, 31);
    const uint32_t dex = dinc - __popc(g), nd = __shfl_sync(0xffffffffu, dinc, 31);
    if (nc < (uint32_t)r || nd == 0) {
        __syncthreads();   // s_flag is rewritten by the next vertex
        return;
    }
    uint16_t* num = reinterpret_cast<uint16_t*>(scratch + nw * kWarpScratch);
    const uint32_t W = (nc + 31) >> 5, Ws = row_stride(W);
    for (uint32_t c = warp_id(); c < runs; c += nw) {
        const uint32_t m = __shfl_sync(0xffffffffu, f, c), dm = __shfl_sync(0xffffffffu, g, c);
        const uint32_t below = (1u << lane) - 1u;
        const uint32_t at = __shfl_sync(0xffffffffu, ex, c) + __popc(m & below);
        const uint32_t dat = __shfl_sync(0xffffffffu, dex, c) + __popc(dm & below);
        if ((m >> lane) & 1u) {
            C[at] = P.wadj[b + c * 32 + lane];
            cnt[at] = 0;
            num[at] = (uint16_t)(((dm >> lane) & 1u) ? dat : nd + at - dat);
        }
    }
    for (uint32_t i = threadIdx.x; i < nc * Ws; i += blockDim.x) rows[i] = 0;
    __syncthreads();
    if (threadIdx.x < nc) bytes += 16 + 4ull * (R.ne[C[threadIdx.x]] - R.nb[C[threadIdx.x]]);
    block_window(C, nc, scratch - kWindowWords);
    __syncthreads();
    block_build_rows(C, nc, W, R.ne, R.adj, R.nb, rows, scratch - kWindowWords, num);
    __syncthreads();
    (void)block_dfs(rows, nc, W, r, cnt, &s_next, scratch, s, S, nd);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nc; i += blockDim.x) {
        const uint32_t j = num[i];
        if (j >= nd || !cnt[j]) continue;
        const uint32_t x = C[i];
        lower(P, x, st_of(P.sl[x]), cnt[j], k, next, next_cnt);
        bytes += 20;
    }
    __syncthreads();
}

// h = 4: the vertices list[0, nv), blocks taking (vertex, slice) units.
// ANY: rows of other lengths are among them and passed over (phase 1 lists
// its vertices by length; a compaction in the same pass may shorten one).
template <bool ANY>
__device__ __forceinline__ void drain_rows(const PeelParams& P, const NPlus& R,
                                           const uint32_t* list, uint32_t nv, uint32_t* grab,
                                           unsigned long long k, uint32_t* next,
                                           uint32_t* next_cnt, uint32_t* smem, uint32_t* s_grab,
                                           unsigned long long& items, unsigned long long& bytes) {
    if (nv == 0) return;
    // as many units as blocks: a slice repeats the row building
    uint32_t S = gridDim.x / nv;
    S = S < 1u ? 1u : (S > kMaxSlices ? kMaxSlices : S);
    for (;;) {
        if (threadIdx.x == 0) *s_grab = atomicAdd(grab, 1u);
        __syncthreads();
        const uint32_t u = *s_grab;
        __syncthreads();
        if (u >= nv * S) break;
        const uint32_t v = list[u / S];
        const uint64_t d = P.wend[v] - P.off[v];
        if (ANY && (d <= kTinyRow || d > kBitmapMax)) continue;
        process_row(P, R, v, u % S, S, k, next, next_cnt, smem, bytes);
        if (threadIdx.x == 0 && u % S == 0) items += d;
    }
}

// P2, phase 1: the cliques destroyed by frontier F (nf vertices, identical
// for every block).  Frontier vertices marked gone (count 0) have no items.
template <int NT, int HC>
__device__ __forceinline__ void process_frontier(
    const PeelParams& P, const NPlus& R, const uint32_t* F, uint32_t nf, unsigned long long k,
    uint32_t* Fnext, uint32_t* next_cnt, uint32_t slot, uint32_t* smem, uint32_t* wC,
    unsigned* wCnt, uint32_t* wRows, unsigned long long* s_pre, unsigned long long* s_red,
    uint32_t* s_grab, uint32_t par, unsigned long long& items, unsigned long long& bytes) {
    const unsigned lane = lane_id();
    const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t gthreads = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t gwarp = gtid >> 5;
    const uint64_t gwarps = gthreads >> 5;
    PeelCtrl* c = P.ctrl;
    if (k == 0) return;   // every frontier vertex has count 0
    if (HC == 2 && nf <= kSmallFront) {
        // flatten (v, neighbour index) items over the whole grid
        block_prefix_degrees<NT>(P, F, nf, s_pre, s_red);
        unsigned long long T = s_pre[nf];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            items += T;
            bytes += 20ull * nf;   // frontier ids and their row bounds
        }
        for (uint64_t t = gtid; t < T; t += gthreads) {
            uint32_t lo = 0, hi = nf;  // last i with s_pre[i] <= t
            while (hi - lo > 1) {
                uint32_t mid = (lo + hi) >> 1;
                if (s_pre[mid] <= t) lo = mid; else hi = mid;
            }
            uint32_t v = F[lo];
            uint32_t u = P.wadj[P.off[v] + (t - s_pre[lo])];
            const uint32_t wu = P.sl[u];
            bool dec;
            (void)cand_ok(wu, u, 0u, v, dec);
            bytes += 4 + 4;
            if (dec) {
                lower(P, u, st_of(wu), 1ull, k, Fnext, next_cnt);
                bytes += 16;
            }
        }
        return;
    }
    if (HC == 2) {
        for (uint64_t i = gwarp; i < nf; i += gwarps) {
            uint32_t v = F[i];
            if (st_of(P.sl[v]) != kFront) continue;
            uint64_t b = P.off[v], e = P.wend[v];
            for (uint64_t p = b + lane; p < e; p += 32) {
                uint32_t u = P.wadj[p];
                const uint32_t wu = P.sl[u];
                bool dec;
                (void)cand_ok(wu, u, 0u, v, dec);
                bytes += 4 + 4;
                if (dec) {
                    lower(P, u, st_of(wu), 1ull, k, Fnext, next_cnt);
                    bytes += 16;
                }
            }
            if (lane == 0) {
                items += e - b;
                bytes += 20;
            }
        }
        return;
    }
    // items spread over every warp of the grid, in batches of kSmallFront
    // vertices: the whole of a small frontier (h = 3, >= 5) or the listed rows
    const bool whole = HC != 4 && nf <= kSmallFront;
    const uint32_t* L = whole ? F : P.heavy;
    const uint32_t nh = whole ? nf : c->hcnt[slot];
    for (uint32_t b0 = 0; b0 < nh; b0 += kSmallFront) {
        const uint32_t nb = nh - b0 < kSmallFront ? nh - b0 : kSmallFront;
        const uint32_t* H = L + b0;
        block_prefix_degrees<NT>(P, H, nb, s_pre, s_red);
        unsigned long long T = s_pre[nb];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            items += T;
            bytes += 20ull * nb;
        }
        for (uint64_t t = gwarp; t < T; t += gwarps) {
            uint32_t lo = 0, hi = nb;
            while (hi - lo > 1) {
                uint32_t mid = (lo + hi) >> 1;
                if (s_pre[mid] <= t) lo = mid; else hi = mid;
            }
            uint32_t v = H[lo];
            uint32_t w = P.wadj[P.off[v] + (t - s_pre[lo])];
            process_vw<HC>(P, R, v, w, k, Fnext, next_cnt, wC, wCnt, wRows, &c->big_cnt[slot],
                       hub_bm_of(P, v, par), bytes);
        }
        __syncthreads();   // s_pre is rewritten by the next batch
    }
    if (whole) return;
    if (HC != 4) {
        // the other vertices: blocks take chunks; in full chunks a warp takes
        // each short row, the block's warps the neighbours of the others
        const uint32_t ch0 = nf / (4u * gridDim.x);
        const uint32_t ch = ch0 < 1u ? 1u : (ch0 > 32u ? 32u : ch0);
        const uint32_t tiny = ch == 32u ? kTinyRow : 0u;
        for (;;) {
            if (threadIdx.x == 0) *s_grab = atomicAdd(&c->grab[slot], ch);
            __syncthreads();
            const uint32_t i0 = *s_grab;
            __syncthreads();
            if (i0 >= nf) break;
            const uint32_t i1 = i0 + ch < nf ? i0 + ch : nf;
            for (uint32_t i = i0 + warp_id(); i < i1; i += NT / 32) {
                const uint32_t v = F[i], wv = P.sl[v];
                if ((wv & kListedBit) || st_of(wv) != kFront) continue;
                const uint64_t d = P.wend[v] - P.off[v];
                if (d > tiny) continue;
                process_tiny<HC>(P, R, v, k, Fnext, next_cnt, wC, wCnt, wRows, bytes);
                if (lane == 0) {
                    items += d;
                    bytes += 24;
                }
            }
            for (uint32_t i = i0; i < i1; i++) {
                const uint32_t v = F[i], wv = P.sl[v];
                if ((wv & kListedBit) || st_of(wv) != kFront) continue;
                const uint64_t b = P.off[v], e = P.wend[v];
                if (e - b <= tiny) continue;
                for (uint64_t p = b + warp_id(); p < e; p += NT / 32)
                    process_vw<HC>(P, R, v, P.wadj[p], k, Fnext, next_cnt, wC, wCnt, wRows,
                               &c->big_cnt[slot], nullptr, bytes);
                if (threadIdx.x == 0) {
                    items += e - b;
                    bytes += 24;
                }
            }
        }
        return;
    }
    // whole neighbourhoods: longer rows first, then the short ones
    drain_rows<false>(P, R, P.vlist, c->vcnt[slot], &c->vgrab[slot], k, Fnext, next_cnt, smem,
                      s_grab, items, bytes);
    __syncthreads();   // the warps' buffers overlap the block's
    const uint32_t ch0 = nf / (8u * (uint32_t)gwarps);
    const uint32_t ch = ch0 < 1u ? 1u : (ch0 > 32u ? 32u : ch0);
    for (;;) {
        uint32_t i0 = 0;
        if (lane == 0) i0 = atomicAdd(&c->grab[slot], ch);
        i0 = __shfl_sync(0xffffffffu, i0, 0);
        if (i0 >= nf) break;
        const uint32_t i1 = i0 + ch < nf ? i0 + ch : nf;
        for (uint32_t i = i0; i < i1; i++) {
            const uint32_t v = F[i], wv = P.sl[v];
            if ((wv & kListedBit) || st_of(wv) != kFront) continue;   // taken above, or none
            process_tiny<HC>(P, R, v, k, Fnext, next_cnt, wC, wCnt, wRows, bytes);
            if (lane == 0) {
                items += P.wend[v] - P.off[v];
                bytes += 24;
            }
        }
    }
}

// P2, phase 1, from round r on: frontiers of at most kSoloFront vertices with
// rows of at most kSoloRow entries, by this block alone, a warp a vertex.  A
// level that leaves along a path has thousands of such rounds; between grid
// barriers each takes 10.6 us (a strip of 3,000 triangles), here 3.1: the loads
// of a vertex's row, of its members' states and of their rows, one after
// another.  Ends when the next frontier is empty, too large or all that is left, when a cascade has
// to be looked at, or after kSoloRounds (the other blocks' waits are bounded).
// F_r is marked on entry; on return F_{r+1} is not, and F_r not retired, as
// at the top of a round (c->solo, c->fcnt).  key, seg, r_end: the band; a
// cascade (multi) ends before round r_end.
template <int NT, int HC>
__device__ __forceinline__ void solo_rounds(const PeelParams& P, const NPlus& R, uint32_t r,
                                            uint32_t f, uint32_t retired, uint32_t rs,
                                            unsigned long long k, bool multi, uint32_t key,
                                            uint32_t seg, uint32_t r_end, uint32_t* wC,
                                            unsigned* wCnt, uint32_t* wRows,
                                            unsigned long long& items,
                                            unsigned long long& bytes) {
    __shared__ uint32_t s_cnt, s_late;
    PeelCtrl* c = P.ctrl;
    const unsigned lane = lane_id(), wid = warp_id();
    const uint64_t t0 = threadIdx.x == 0 ? globaltimer_ns() : 0;
    if (threadIdx.x == 0) s_cnt = s_late = 0;
    __syncthreads();
    for (uint32_t step = 1;; step++) {
        const uint32_t* F = P.front[r % 3];
        uint32_t* N = P.front[(r + 1) % 3];
        for (uint32_t i = wid; i < f; i += NT / 32) {
            const uint32_t v = F[i];
            if (st_of(P.sl[v]) != kFront) continue;
            process_tiny<HC, true>(P, R, v, k, N, &s_cnt, wC, wCnt, wRows, bytes);
            if (lane == 0) {
                items += P.wend[v] - P.off[v];
                bytes += 24;
            }
        }
        if (threadIdx.x == 0 && (step & 15u) == 0 && globaltimer_ns() - t0 > P.wait_ns / 4)
            s_late = 1;
        __syncthreads();
        const uint32_t fn = s_cnt;
        bool stop = fn == 0 || fn > kSoloFront || step == kSoloRounds || s_late ||
                    retired + f + fn == P.n ||
                    (multi && (retired + f - seg + fn > kBandMax || r + 1 >= r_end));
        unsigned long long d = 1;
        if (threadIdx.x < fn && !stop) {
            const uint32_t v = N[threadIdx.x];
            d = P.deg[v];
            if (P.wend[v] - P.off[v] > kSoloRow) stop = true;
        }
        if (__syncthreads_or(stop)) {
            if (threadIdx.x == 0) {
                c->fcnt[r % 3] = f;
                c->fcnt[(r + 1) % 3] = fn;
                c->solo[0] = r + 1;
                c->solo[1] = retired;
                c->solo[2] = rs;
                // the counters by round, which no round in between has cleared
                for (int i = 0; i < 3; i++)
                    c->hcnt[i] = c->vcnt[i] = c->vgrab[i] = c->grab[i] = c->lrow[i] = 0;
                for (int i = 0; i < 6; i++) c->big_cnt[i] = c->bgrab[i] = 0;
            }
            return;
        }
        // retire F_r, mark F_{r+1}
        unsigned long long gone = 0;
        if (threadIdx.x < f) {
            const uint32_t v = F[threadIdx.x];
            gone = P.deg[v];
            P.sl[v] = kGone;
            P.band_of[v] = key;
            P.mem[retired + threadIdx.x] = v;
            if (!multi) {
                P.core[v] = k;
                if (P.rnd) P.rnd[v] = rs;
            }
            bytes += 4 + 4 + 8 + 8 + 4 + (P.rnd ? 4 : 0);
        }
        if (wid < (kSoloFront + 31) / 32) {
            gone = warp_sum(gone);
            if (lane == 0 && gone) atomicAdd(&c->destroyed, gone);
        }
        if (threadIdx.x < fn) {
            P.sl[N[threadIdx.x]] = d ? kFront : kGone;
            bytes += 4 + 4 + 8 + 16;
        }
        retired += f;
        if (!multi) rs++;
        f = fn;
        r++;
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
    }
}

// P2, phase 2: the frontiers of all bands together (nf vertices), in batches
// whose items are flattened over the grid.
template <int NT, int HC>
__device__ __forceinline__ void process_bands(
    const PeelParams& P, const NPlus& R, const uint32_t* F, uint32_t nf, uint32_t slot,
    uint32_t* smem, uint32_t* wC, unsigned* wCnt, uint32_t* wRows, unsigned long long* s_pre,
    unsigned long long* s_red, uint32_t* s_grab, unsigned long long& items,
    unsigned long long& bytes) {
    PeelCtrl* c = P.ctrl;
    const unsigned lane = lane_id();
    const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t gthreads = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t gwarp = gtid >> 5;
    const uint64_t gwarps = gthreads >> 5;
    for (uint32_t b0 = 0; b0 < nf; b0 += kSmallFront) {
        const uint32_t nb = nf - b0 < kSmallFront ? nf - b0 : kSmallFront;
        const uint32_t* H = F + b0;
        // h = 4: only the rows that are not taken whole below
        block_prefix_degrees<NT>(P, H, nb, s_pre, s_red, HC == 4 ? kBitmapMax : 0u);
        const unsigned long long T = s_pre[nb];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            items += T;
            bytes += 20ull * nb;
        }
        // the frontier vertex of item t: last i with s_pre[i] <= t
        auto at = [&](uint64_t t) -> uint32_t {
            uint32_t lo = 0, hi = nb;
            while (hi - lo > 1) {
                uint32_t mid = (lo + hi) >> 1;
                if (s_pre[mid] <= t) lo = mid; else hi = mid;
            }
            return lo;
        };
        if (HC == 2) {
            for (uint64_t t = gtid; t < T; t += gthreads) {
                const uint32_t i = at(t), v = H[i];
                const uint32_t u = P.wadj[P.off[v] + (t - s_pre[i])];
                bool dec;
                (void)cand_ok(P.sl[u], u, P.sl[v] >> kKeyShift, v, dec);
                bytes += 4 + 4;
                if (dec) {
                    atomic_sub_u64(&P.deg[u], 1ull);
                    bytes += 16;
                }
            }
        } else if (HC == 3) {
            // a warp looks at up to 32 items at once, one a lane, and takes the
            // pairs among them one by one: most items name a vertex of a
            // later band and need nothing more.  A lane's items lie gwarps
            // apart: members of one band are neighbours in a row, and taken
            // in runs they fell to a few warps
            for (uint64_t t0 = gwarp; t0 < T; t0 += gwarps * 32) {
                const uint64_t t = t0 + lane * gwarps;
                uint32_t v = 0, u = 0, kv = 0;
                bool dec = false;
                if (t < T) {
                    const uint32_t i = at(t);
                    v = H[i];
                    u = P.wadj[P.off[v] + (t - s_pre[i])];
                    kv = P.sl[v] >> kKeyShift;
                    (void)cand_ok(P.sl[u], u, kv, v, dec);
                    bytes += 4 + 4;
                }
                unsigned todo = __ballot_sync(0xffffffffu, dec);
                while (todo) {
                    const int l = __ffs(todo) - 1;
                    todo &= todo - 1;
                    process_pair(P, __shfl_sync(0xffffffffu, v, l),
                                 __shfl_sync(0xffffffffu, kv, l),
                                 __shfl_sync(0xffffffffu, u, l), bytes);
                }
            }
        } else {
            for (uint64_t t = gwarp; t < T; t += gwarps) {
                const uint32_t i = at(t), v = H[i];
                const uint32_t w = P.wadj[P.off[v] + (t - s_pre[i])];
                process_vw<HC>(P, R, v, w, 0ull, nullptr, nullptr, wC, wCnt, wRows,
                           &c->big_cnt[slot], nullptr, bytes);
            }
        }
        __syncthreads();   // s_pre is rewritten by the next batch
    }
    if (HC != 4) return;
    drain_rows<true>(P, R, F, nf, &c->vgrab[slot], 0ull, nullptr, nullptr, smem, s_grab, items,
                     bytes);
    __syncthreads();   // the warps' buffers overlap the block's
    for (uint64_t i = gwarp; i < nf; i += gwarps) {
        const uint32_t v = F[i];
        const uint64_t d = P.wend[v] - P.off[v];
        if (d > kTinyRow) continue;
        process_tiny<HC>(P, R, v, 0ull, nullptr, nullptr, wC, wCnt, wRows, bytes);
        if (lane == 0) items += d;
    }
}

// P2b: the round's mid items (warp groups) and big items (blocks).
template <int NT>
__device__ __forceinline__ void process_queued(const PeelParams& P, const NPlus& R, uint32_t slot,
                                               uint32_t nb, uint32_t nm, unsigned long long k,
                                               uint32_t* next, uint32_t* next_cnt, uint32_t* smem,
                                               bool hubs, uint32_t par, uint32_t* s_grab,
                                               unsigned long long& bytes) {
    PeelCtrl* c = P.ctrl;
    if (nb > P.big_cap) nb = (uint32_t)P.big_cap;
    if (nm > P.mid_cap) nm = P.mid_cap;
    if (nm) {
        drain_mid<NT>(P, R, nm, &c->bgrab[3 + slot], k, next, next_cnt, bytes);
        __syncthreads();
    }
    for (;;) {
        if (threadIdx.x == 0) *s_grab = atomicAdd(&c->bgrab[slot], 1u);
        __syncthreads();
        const uint32_t i = *s_grab;
        __syncthreads();
        if (i >= nb) break;
        const uint2 it = P.big[i];
        process_big(P, R, it.x, it.y, k, next, next_cnt, smem,
                    hubs ? hub_bm_of(P, it.x, par) : nullptr, bytes);
    }
}

// ---------------------------------------------------------------- kernel
// HC: the clique size, 5 for all from 5 on (P.h): each has its own registers.
template <int NT, int HC>
__global__ void __launch_bounds__(NT, 1024 / NT) k_peel(PeelParams P) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ unsigned long long s_pre[kSmallFront + 1];
    __shared__ unsigned long long s_red[NW];
    __shared__ uint32_t s_hist[kBins];
    __shared__ uint32_t s_wtot[NW];
    __shared__ unsigned long long s_bmin[2][NW], s_bsum[2][NW];
    __shared__ uint32_t s_bcnt[2][NW], s_bleft[2][NW];
    __shared__ uint32_t s_n;
    __shared__ uint32_t s_grab;
    PeelCtrl* c = P.ctrl;
    const unsigned lane = lane_id(), wid = warp_id();
    const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t gthreads = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t gwarp = gtid >> 5;
    const uint64_t gwarps = gthreads >> 5;
    uint32_t* wC = smem + (size_t)wid * kWarpWords;
    unsigned* wCnt = wC + kWarpCand;
    uint32_t* wRows = wC + 2 * kWarpCand;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    const NPlus R1{P.wadj, P.wnb, P.wend};
    const NPlus R2{P.nadj, P.nsplit, P.off + 1};

    unsigned long long k = P.k0;           // level floor (threshold pruning when > 0)
    unsigned long long klow = k;           // k before the last jump
    uint32_t r = 0, jumps = 0, nbar = 0, ncompact = 0;
    int ap = 0;
    uint32_t alive_cnt = P.n;              // entries of the alive list
    uint32_t compacted_at = P.n;           // alive count at the last row compaction
    uint32_t retired = 0;                  // vertices in mem
    uint32_t nb = 0;                       // multi-level bands so far
    bool multi = false;                    // the current band has several levels
    uint32_t seg = 0;                      // where it starts in mem
    uint32_t rjump = 0;                    //   and its first round
    uint32_t fails = 0, hold = 0;          // cascades undone in a row; jumps without bands
    unsigned long long gone0 = 0;          // lead: cliques destroyed before the band
    uint32_t rs = 0;                       // rounds of single-level bands so far
    unsigned long long items = 0, bytes = 0, waited = 0;

    // Block 0's time per phase (thread 0, %globaltimer); the time inside
    // barriers is counted separately in `waited`.
    __shared__ unsigned long long tph[8];
    if (threadIdx.x < 8) tph[threadIdx.x] = 0;
    uint64_t tlast = lead ? globaltimer_ns() : 0;
#define PHASE(i)                                 \
    do {                                         \
        if (lead) {                              \
            uint64_t t_ = globaltimer_ns();      \
            tph[i] += t_ - tlast;                \
            tlast = t_;                          \
        }                                        \
    } while (0)
#define BARRIER(i)                                         \
    do {                                                   \
        PHASE(i);                                          \
        nbar++;                                            \
        if (!grid_barrier(c, P.wait_ns, waited)) goto out; \
        if (lead) tlast = globaltimer_ns();                \
    } while (0)

    // ============================================================ phase 1
    for (;;) {
        // ---------------------------------------------------------- P1
        const uint32_t fprev = r ? c->fcnt[(r + 2) % 3] : 0u;
        if (fprev) {
            const uint32_t* Fprev = P.front[(r + 2) % 3];
            const uint32_t key = 2u * nb - (multi ? 1u : 0u);
            unsigned long long gone = 0;
            for (uint64_t i = gtid; i < fprev; i += gthreads) {
                uint32_t v = Fprev[i];
                gone += P.deg[v];
                P.sl[v] = kGone;
                P.band_of[v] = key;
                P.mem[retired + i] = v;
                if (!multi) {
                    P.core[v] = k;
                    if (P.rnd) P.rnd[v] = rs;
                }
                bytes += 4 + 4 + 8 + 8 + 4 + (P.rnd ? 4 : 0);
            }
            gone = warp_sum(gone);
            if (lane == 0 && gone) atomicAdd(&c->destroyed, gone);
            retired += fprev;
            if (!multi) rs++;
        }
        uint32_t fcur = c->fcnt[r % 3];
        uint32_t* Fcur = P.front[r % 3];
        const bool undo = multi && (retired - seg + fcur > kBandMax ||
                                    (fcur && r - rjump >= kBandRounds));
        // the bitmaps of F_{r-1}'s hubs are zeroed for round r+1
        if (r && P.hub_slots) {
            uint32_t nhub = c->hubcnt[(r + 1) & 1];
            if (nhub > P.hub_slots) nhub = P.hub_slots;
            if (nhub) hub_bitmaps<NT>(P, nhub, (r + 1) & 1, true, s_pre, s_red, bytes);
        }
        // mark F_r; all but the short rows are also listed
        for (uint64_t base = gwarp * 32; base < fcur && !undo; base += gwarps * 32) {
            uint64_t i = base + lane;
            uint32_t v = 0, cls = 0;
            bool lrow = false;
            if (i < fcur) {
                v = Fcur[i];
                P.sl[v] = front_word<HC>(P, c, v, r & 1, cls, lrow);
                bytes += 4 + 4 + 8 + (HC > 2 ? 16 : 0);
            }
            if (HC > 2) {
                warp_append(cls == 2, v, &c->hcnt[r % 3], P.heavy);
                warp_append(cls == 1, v, &c->vcnt[r % 3], P.vlist);
                if (fcur <= kSoloFront && __any_sync(0xffffffffu, lrow) && lane == 0)
                    c->lrow[r % 3] = 1;
            }
        }
        if (lead) {
            if (r) {
                c->big_cnt[(r + 2) % 3] = 0;
                c->bgrab[(r + 2) % 3] = 0;
                c->big_cnt[3 + (r + 2) % 3] = 0;
                c->bgrab[3 + (r + 2) % 3] = 0;
            }
            c->fcnt[(r + 1) % 3] = 0;
            c->hcnt[(r + 1) % 3] = 0;
            c->lrow[(r + 1) % 3] = 0;
            c->vcnt[(r + 1) % 3] = 0;
            c->vgrab[(r + 1) % 3] = 0;
            c->grab[(r + 1) % 3] = 0;
        }
        BARRIER(0);
        if (undo) {
            // back to the band's start; its first level goes alone, as do the
            // levels of the next 2^fails - 1 jumps
            for (uint64_t i = gtid; i < alive_cnt; i += gthreads) {
                const uint32_t v = P.alive[ap][i];
                P.deg[v] = P.c0[v];
                P.sl[v] = kAlive;
                bytes += 4 + 16 + 4;
            }
            if (lead) {
                c->fcnt[r % 3] = 0;
                c->destroyed = gone0;
            }
            fcur = 0;
            retired = seg;
            nb--;
            multi = false;
            k = klow;
            fails = fails < 10 ? fails + 1 : 10;
            hold = 1u << (fails - 1);
            BARRIER(0);
        }

        // ------------------------------------------------------ band jump
        if (fcur == 0) {
            const uint32_t left = P.n - retired;
            if (left == 0) break;
            if (multi) fails = 0;
            const bool banding = left <= P.band_max && nb < kMaxBands && hold == 0 &&
                                 (HC > 2 || rs >= kBandAfter2);
            if (hold) hold--;
            const uint32_t* Ain = P.alive[ap];
            uint32_t* Aout = P.alive[ap ^ 1];
            uint32_t* ghist = c->hist[jumps & 1];
            unsigned long long mn = ~0ull;
            if (banding) {
                for (uint32_t i = threadIdx.x; i < kBins; i += NT) s_hist[i] = 0;
                if (lead && c->band_n == 0) {
                    c->band_n = left;
                    c->band_round = r;
                }
                __syncthreads();
            }
            for (uint64_t base = gwarp * 32; base < alive_cnt; base += gwarps * 32) {
                uint64_t i = base + lane;
                bool keep = false;
                uint32_t v = 0;
                if (i < alive_cnt) {
                    v = Ain[i];
                    bytes += 4 + 4;
                    if (st_of(P.sl[v]) != kGone) {
                        keep = true;
                        unsigned long long d = P.deg[v];
                        mn = d < mn ? d : mn;
                        if (P.snap) P.snap[v] = d;
                        if (banding) {
                            P.c0[v] = d;
                            atomicAdd(&s_hist[d > k ? bin_of(d - k - 1) : 0u], 1u);
                            bytes += 8;
                        }
                        bytes += 8 + 4;
                    }
                }
                warp_append(keep, v, &c->new_alive[jumps & 1], Aout);
            }
            mn = warp_min_u64(mn);
            if (lane == 0 && mn != ~0ull) atomicMin(&c->min_deg[jumps & 1], mn);
            if (banding) {
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < kBins; i += NT)
                    if (s_hist[i]) atomicAdd(&ghist[i], s_hist[i]);
            }
            BARRIER(1);
            ap ^= 1;
            alive_cnt = left;
            const unsigned long long m2 = c->min_deg[jumps & 1];
            const unsigned long long kmin = m2 > k ? m2 : k;
            multi = false;
            klow = k;
            seg = retired;
            rjump = r;
            unsigned long long kt = 0;
            if (banding && m2 > k) {
                const uint32_t tmax = band_aim(left);
                kt = pick_threshold<NT>(ghist, k, tmax, tmax / 8, s_wtot, &s_n);
                multi = kt > m2;
            }
            if (lead) {
                gone0 = c->destroyed;
                const unsigned long long mu = P.mu0 - gone0;
                if (multi) {
                    Band& b = P.bands[nb];
                    b.k = k;
                    b.mu = mu;
                    b.seg = retired;
                    b.rbase = rs;
                    b.nlev = 0;
                    b.rounds = 0;
                } else {
                    P.t_k[retired] = kmin;
                    P.t_size[retired] = left;
                    P.t_mu[retired] = mu;
                }
                c->min_deg[(jumps + 1) & 1] = ~0ull;
                c->new_alive[(jumps + 1) & 1] = 0;
            }
            if (blockIdx.x == gridDim.x - 1 && P.band_max)
                for (uint32_t i = threadIdx.x; i < kBins; i += NT) c->hist[(jumps + 1) & 1][i] = 0;
            if (multi) nb++;
            k = multi ? kt : kmin;
            jumps++;
            // Rows may be compacted in this same phase: compaction keeps
            // every vertex that is not removed, whether or not it is being
            // marked frontier concurrently (a frontier vertex of count 0 is
            // marked gone, but lies in no clique).
            if (P.compact && 2ull * left <= compacted_at) {
                compacted_at = left;
                ncompact++;
                for (uint64_t i = gwarp; i < left; i += gwarps) compact_row(P, Aout[i], 0u, bytes);
            }
            for (uint64_t base = gwarp * 32; base < left; base += gwarps * 32) {
                uint64_t i = base + lane;
                bool in = false, lrow = false;
                uint32_t v = 0, cls = 0;
                if (i < left) {
                    v = Aout[i];
                    bytes += 4 + 8;
                    if (P.deg[v] <= k) {
                        in = true;
                        P.sl[v] = front_word<HC>(P, c, v, r & 1, cls, lrow);
                        bytes += 4 + 4 + (HC > 2 ? 16 : 0);
                    }
                }
                warp_append(in, v, &c->fcnt[r % 3], Fcur);
                if (HC > 2) {
                    warp_append(cls == 2, v, &c->hcnt[r % 3], P.heavy);
                    warp_append(cls == 1, v, &c->vcnt[r % 3], P.vlist);
                    if (__any_sync(0xffffffffu, lrow) && lane == 0) c->lrow[r % 3] = 1;
                }
            }
            BARRIER(2);
            fcur = c->fcnt[r % 3];
        }
        // ---------------------------------------------------------- P2
        if (P.hub_slots) {
            uint32_t nhub = c->hubcnt[r & 1];
            if (nhub > P.hub_slots) nhub = P.hub_slots;
            if (lead) c->hubcnt[(r + 1) & 1] = 0;   // read last in this round's P1
            if (nhub) {
                hub_bitmaps<NT>(P, nhub, r & 1, false, s_pre, s_red, bytes);
                BARRIER(3);
            }
        }
        if (HC > 2 && r - rjump >= kSoloAfter && fcur <= kSoloFront && k > 0 &&
            retired + fcur < P.n && !c->lrow[r % 3]) {
            if (blockIdx.x == 0)
                solo_rounds<NT, HC>(P, R1, r, fcur, retired, rs, k, multi,
                                    2u * nb - (multi ? 1u : 0u), seg, rjump + kBandRounds, wC,
                                    wCnt, wRows, items, bytes);
            BARRIER(3);
            r = *(volatile uint32_t*)&c->solo[0];
            retired = *(volatile uint32_t*)&c->solo[1];
            rs = *(volatile uint32_t*)&c->solo[2];
            continue;
        }
        // when everything left leaves at once there is no count to lower
        if (retired + fcur < P.n) {
            process_frontier<NT, HC>(P, R1, Fcur, fcur, k, P.front[(r + 1) % 3],
                                 &c->fcnt[(r + 1) % 3], r % 3, smem, wC, wCnt, wRows, s_pre,
                                 s_red, &s_grab, r & 1, items, bytes);
            BARRIER(3);
            if (HC >= 4 && P.big_cap) {
                const uint32_t nbig = c->big_cnt[r % 3], nmid = c->big_cnt[3 + r % 3];
                if (nbig || nmid) {
                    process_queued<NT>(P, R1, r % 3, nbig, nmid, k, P.front[(r + 1) % 3],
                                       &c->fcnt[(r + 1) % 3], smem, true, r & 1, &s_grab, bytes);
                    BARRIER(3);
                }
            }
        }
        r++;
    }

    // ============================================================ phase 2
    if (nb) {
        const uint64_t t2 = lead ? globaltimer_ns() : 0;
        // every vertex gets its key; members of multi-level bands are alive
        // again with their count at the band's start
        // (earlier vertices keep key 0, below every band's)
        const uint32_t first = P.bands[0].seg;
        for (uint64_t i = first + gtid; i < P.n; i += gthreads) {
            const uint32_t v = P.mem[i], key = P.band_of[v];
            if (key & 1u) P.deg[v] = P.c0[v];
            P.sl[v] = (key << kKeyShift) | ((key & 1u) ? kAlive : kGone);
            bytes += 4 + 4 + 4 + 16;
        }
        if (lead) {
            c->fcnt[0] = c->fcnt[1] = c->fcnt[2] = 0;
            c->busy[0] = c->busy[1] = c->busy[2] = 0;
            c->vgrab[0] = c->vgrab[1] = c->vgrab[2] = 0;
            for (int i = 0; i < 6; i++) c->big_cnt[i] = c->bgrab[i] = 0;
        }
        // band sizes: the first position past seg whose key differs
        for (uint64_t i = first + gtid; i < P.n; i += gthreads) {
            const uint32_t key = P.band_of[P.mem[i]];
            if ((key & 1u) && (i + 1 == P.n || P.band_of[P.mem[i + 1]] != key)) {
                Band& b = P.bands[key >> 1];
                b.size = b.left = (uint32_t)(i + 1) - b.seg;
                b.above = P.n - (uint32_t)(i + 1);
            }
        }
        BARRIER(4);
        // rows of the members without earlier bands
        for (uint64_t i = first + gwarp; i < P.n; i += gwarps) {
            const uint32_t v = P.mem[i], key = P.sl[v] >> kKeyShift;
            if (key & 1u) compact_row(P, v, key, bytes);
        }
        BARRIER(5);
        uint32_t q = 0;   // round
        uint32_t flip = 0;
        for (;;) {
            // ------------------------------------------------------- A
            uint32_t* F = P.front[q & 1];
            uint32_t* fcnt = &c->fcnt[q % 3];
            for (uint32_t bi = blockIdx.x; bi < nb; bi += gridDim.x) {
                Band& B = P.bands[bi];
                const uint32_t left = B.left;
                if (left == 0) continue;
                const uint32_t seg = B.seg;
                const unsigned long long bk = B.k;
                const uint32_t rb = B.rounds;
                // retire the frontier; least count, members at <= k and
                // members left
                unsigned long long mn = ~0ull, sum = 0;
                uint32_t cnt = 0, al = 0;
                uint32_t v0 = 0, w0 = kGone;      // this thread's first member
                unsigned long long d0 = 0;
                for (uint32_t i = threadIdx.x; i < left; i += NT) {
                    const uint32_t v = P.mem[seg + i];
                    uint32_t w = P.sl[v];
                    unsigned long long d = 0;
                    if (st_of(w) != kGone) {
                        d = P.deg[v];
                        if (st_of(w) == kFront) {
                            sum += d;
                            P.core[v] = bk;
                            if (P.rnd) P.rnd[v] = rb - 1;
                            w = (w & ~3u) | kGone;
                            P.sl[v] = w;
                            bytes += 12;
                        } else {
                            al++;
                            cnt += d <= bk;
                            mn = d < mn ? d : mn;
                        }
                        bytes += 8;
                    }
                    bytes += 8;
                    if (i < NT) {
                        v0 = v;
                        w0 = w;
                        d0 = d;
                    }
                }
                mn = warp_min_u64(mn);
                sum = warp_sum(sum);
                cnt = __reduce_add_sync(0xffffffffu, cnt);
                al = __reduce_add_sync(0xffffffffu, al);
                if (lane == 0) {
                    s_bmin[flip][wid] = mn;
                    s_bsum[flip][wid] = sum;
                    s_bcnt[flip][wid] = cnt;
                    s_bleft[flip][wid] = al;
                }
                __syncthreads();
                mn = warp_min_u64(lane < NW ? s_bmin[flip][lane] : ~0ull);
                sum = warp_sum(lane < NW ? s_bsum[flip][lane] : 0ull);
                cnt = __reduce_add_sync(0xffffffffu, lane < NW ? s_bcnt[flip][lane] : 0u);
                al = __reduce_add_sync(0xffffffffu, lane < NW ? s_bleft[flip][lane] : 0u);
                flip ^= 1;
                const unsigned long long mu = B.mu - sum;
                unsigned long long kk = bk;
                const bool jump = cnt == 0;
                if (jump && al) {
                    kk = mn > bk ? mn : bk;
                    if (P.snap)
                        for (uint32_t i = threadIdx.x; i < left; i += NT) {
                            const uint32_t v = P.mem[seg + i];
                            if (st_of(P.sl[v]) == kAlive) P.snap[v] = P.deg[v];
                        }
                }
                // mark the next frontier; members of count 0 lie in no clique and
                // have nothing to enumerate
                for (uint32_t b0 = 0; b0 < left; b0 += NT) {
                    const uint32_t i = b0 + threadIdx.x;
                    uint32_t v = v0, w = w0;
                    unsigned long long d = d0;
                    if (b0) {
                        w = kGone;
                        if (i < left) {
                            v = P.mem[seg + i];
                            w = P.sl[v];
                            d = P.deg[v];
                        }
                    }
                    const bool in = i < left && st_of(w) == kAlive && d <= kk;
                    if (in) P.sl[v] = (w & ~3u) | kFront;
                    warp_append(in && d, v, fcnt, F);
                }
                __syncthreads();   // every thread has read the band's record
                if (threadIdx.x == 0) {
                    B.mu = mu;
                    if (al) {
                        atomicAdd(&c->busy[q % 3], 1u);
                        B.rounds = rb + 1;
                        if (jump) {
                            const uint32_t at = seg + B.nlev;
                            P.t_k[at] = kk;
                            P.t_size[at] = B.above + al;
                            P.t_mu[at] = mu;
                            B.nlev++;
                            B.k = kk;
                        }
                    } else {
                        B.left = 0;
                    }
                }
            }
            if (lead) {
                c->fcnt[(q + 1) % 3] = 0;
                c->busy[(q + 1) % 3] = 0;
                c->vgrab[(q + 1) % 3] = 0;
                if (q) {
                    c->big_cnt[(q + 2) % 3] = 0;
                    c->bgrab[(q + 2) % 3] = 0;
                    c->big_cnt[3 + (q + 2) % 3] = 0;
                    c->bgrab[3 + (q + 2) % 3] = 0;
                }
            }
            BARRIER(4);
            if (c->busy[q % 3] == 0) break;
            // ------------------------------------------------------- P2
            process_bands<NT, HC>(P, R2, F, *fcnt, q % 3, smem, wC, wCnt, wRows, s_pre, s_red,
                              &s_grab, items, bytes);
            BARRIER(6);
            if (HC >= 4 && P.big_cap) {
                const uint32_t nbig = c->big_cnt[q % 3], nmid = c->big_cnt[3 + q % 3];
                if (nbig || nmid) {
                    process_queued<NT>(P, R2, q % 3, nbig, nmid, 0ull, nullptr, nullptr, smem,
                                       false, 0, &s_grab, bytes);
                    BARRIER(7);
                }
            }
            q++;
        }
        if (lead) c->phase2_ns = globaltimer_ns() - t2;
        r += q;
    }
    // ======================================================== final pass
    // level records in order (their positions ascend), and the removal
    // rounds: a band's rounds start after those of the bands before it
    {
        uint32_t run = 0;
        for (uint32_t b0 = 0; b0 < nb; b0 += NT) {
            const uint32_t i = b0 + threadIdx.x;
            const uint32_t x = i < nb ? P.bands[i].rounds : 0u;
            uint32_t tot;
            const uint32_t at = block_scan_count<NT>(x, s_wtot, &tot);
            if (blockIdx.x == 0 && i < nb) P.bands[i].size = run + at;   // size is free now
            run += tot;
        }
        const uint32_t lo = (uint32_t)((uint64_t)P.n * blockIdx.x / gridDim.x);
        const uint32_t hi = (uint32_t)((uint64_t)P.n * (blockIdx.x + 1) / gridDim.x);
        uint32_t mine = 0;
        for (uint32_t i = lo + threadIdx.x; i < hi; i += NT) mine += P.t_size[i] != 0;
        uint32_t tot;
        (void)block_scan_count<NT>(mine, s_wtot, &tot);
        if (threadIdx.x == 0) P.blkcnt[blockIdx.x] = tot;
        BARRIER(0);
        if (P.rnd && nb) {
            const uint32_t tail = run;
            for (uint64_t i = gtid; i < P.n; i += gthreads) {
                const uint32_t key = P.band_of[i], j = key >> 1;
                uint32_t add = j < nb ? P.bands[j].size : tail;
                if (key & 1u) add += P.bands[j].rbase;
                P.rnd[i] += add;
            }
        }
        uint32_t before = 0, all = 0;
        for (uint32_t t = threadIdx.x; t < gridDim.x; t += NT) {
            const uint32_t x = P.blkcnt[t];
            all += x;
            before += t < blockIdx.x ? x : 0u;
        }
        uint32_t base, nlev;
        (void)block_scan_count<NT>(before, s_wtot, &base);
        (void)block_scan_count<NT>(all, s_wtot, &nlev);
        for (uint32_t b0 = lo; b0 < hi; b0 += NT) {
            const uint32_t i = b0 + threadIdx.x;
            const uint32_t sz = i < hi ? P.t_size[i] : 0u;
            const uint32_t at = base + block_scan_count<NT>(sz ? 1u : 0u, s_wtot, &tot);
            if (sz) {
                P.lvl_k[at] = P.t_k[i];
                P.lvl_size[at] = sz;
                P.lvl_mu[at] = P.t_mu[i];
                if (at + 1 == nlev) c->kmax = P.t_k[i];
            }
            base += tot;
        }
        if (lead) {
            c->nlevels = nlev;
            c->rounds = rs + run;
        }
    }
out:
#undef BARRIER
#undef PHASE
    if (lead) {
        for (int i = 0; i < 8; i++) c->tph[i] = tph[i];
        c->nbands = nb;
        c->grid_rounds = r;
        c->barrier_ns = waited;
        c->barriers = nbar;
        c->compactions = ncompact;
    }
    items = warp_sum(items);
    bytes = warp_sum(bytes);
    if (lane == 0 && items) atomicAdd(&c->items, items);
    if (lane == 0 && bytes) atomicAdd(&c->bytes, bytes);
}

// The h = 2 peel of a small graph by one block: every count, row start and
// state in shared memory, so that a round is a few block barriers and one
// trip to the rows (L2) instead of grid barriers and global bookkeeping.
// `order` lists the vertices as they leave: F_r is order[a, b), F_{r+1} is
// appended behind it.  stamp[v] is the round v leaves in (kStay while alive),
// so a vertex is a frontier member in that round and gone after it without
// being marked; the thread whose decrement takes a count to k appends the
// vertex.  Frontier members of larger id are lowered too: what is left of a
// frontier member's count is the number of edges credited to it.
// Bound by the latency of a round (block scan, row load, shared atomics).
struct Peel2Block {
    uint32_t n;
    const uint64_t* off;
    const uint32_t* adj;
    uint64_t* core;
    uint32_t* rnd;
    uint64_t* lvl_k;
    uint32_t* lvl_size;
    uint64_t* lvl_mu;
    PeelCtrl* ctrl;
    unsigned long long mu0;
    uint32_t k0;
};

constexpr size_t peel2_block_smem(uint32_t n) { return (size_t)n * 12 + 16; }

__global__ void __launch_bounds__(1024, 1) k_peel2_block(Peel2Block P) {
    constexpr int NT = 1024, NW = NT / 32;
    constexpr uint32_t kStay = 0xffffu;   // rounds stay below n <= kOneBlockN
    extern __shared__ __align__(16) uint32_t smem[];
    uint32_t* deg = smem;                                  // [n]
    uint32_t* at = deg + P.n;                              // [n + 1] row starts
    uint16_t* stamp = (uint16_t*)(at + P.n + 1);           // [n]
    uint16_t* order = stamp + P.n;                         // [n]
    __shared__ uint32_t s_pre[NT];
    __shared__ uint32_t s_wtot[NW];
    __shared__ uint32_t s_min[NW];
    __shared__ unsigned long long s_sum[NW];
    __shared__ uint32_t s_end;
    const uint32_t n = P.n, tid = threadIdx.x;
    const unsigned lane = lane_id(), wid = warp_id();
    for (uint32_t v = tid; v <= n; v += NT) at[v] = (uint32_t)P.off[v];
    __syncthreads();
    for (uint32_t v = tid; v < n; v += NT) {
        deg[v] = at[v + 1] - at[v];
        stamp[v] = (uint16_t)kStay;
    }
    if (tid == 0) s_end = 0;
    __syncthreads();
    uint32_t a = 0, b = 0;          // F_r = order[a, b)
    uint32_t r = 0, k = P.k0, nlev = 0;
    unsigned long long mu = P.mu0, gone = 0;   // gone: this thread's share since the last level
    unsigned long long items = 0;
    for (;;) {
        if (a == b) {
            // a new level: k = max(k, least count left), recorded before its
            // first round
            if (a == n) break;
            uint32_t mn = 0xffffffffu;
            for (uint32_t v = tid; v < n; v += NT)
                if (stamp[v] == kStay) mn = min(mn, deg[v]);
            mn = __reduce_min_sync(0xffffffffu, mn);
            gone = warp_sum(gone);
            if (lane == 0) {
                s_min[wid] = mn;
                s_sum[wid] = gone;
            }
            gone = 0;
            __syncthreads();
            mn = __reduce_min_sync(0xffffffffu, s_min[lane]);
            mu -= warp_sum(s_sum[lane]);
            k = mn > k ? mn : k;
            if (tid == 0) {
                P.lvl_k[nlev] = k;
                P.lvl_size[nlev] = n - a;
                P.lvl_mu[nlev] = mu;
            }
            nlev++;
            for (uint32_t v0 = 0; v0 < n; v0 += NT) {
                const uint32_t v = v0 + tid;
                const bool in = v < n && stamp[v] == kStay && deg[v] <= k;
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                if (!bal) continue;
                uint32_t base = 0;
                if (lane == 0) base = atomicAdd(&s_end, (uint32_t)__popc(bal));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (in) {
                    order[base + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)v;
                    stamp[v] = (uint16_t)r;
                }
            }
            __syncthreads();
            b = s_end;
        }
        // the rows of F_r, flattened over the block, NT frontier vertices at
        // a time
        for (uint32_t f0 = a; f0 < b; f0 += NT) {
            const uint32_t i = f0 + tid;
            uint32_t d = 0;
            if (i < b) {
                const uint32_t v = order[i];
                d = at[v + 1] - at[v];
                P.core[v] = k;
                if (P.rnd) P.rnd[v] = r;
            }
            uint32_t T;
            const uint32_t ex = block_scan_count<NT>(d, s_wtot, &T);
            s_pre[tid] = ex;   // entries past the frontier hold T
            __syncthreads();
            if (tid == 0) items += T;
            const uint32_t nb = b - f0 < NT ? b - f0 : NT;
            for (uint32_t t = tid; t < T; t += NT) {
                uint32_t lo = 0, hi = nb;   // last j with s_pre[j] <= t
                while (hi - lo > 1) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (s_pre[mid] <= t) lo = mid; else hi = mid;
                }
                const uint32_t v = order[f0 + lo];
                const uint32_t u = P.adj[at[v] + (t - s_pre[lo])];
                const uint32_t su = stamp[u];
                if (su > r) {
                    // alive (perhaps already queued for the next round)
                    if (atomicSub(&deg[u], 1u) == k + 1u) {
                        order[atomicAdd(&s_end, 1u)] = (uint16_t)u;
                        stamp[u] = (uint16_t)(r + 1u);
                    }
                } else if (su == r && u > v) {
                    atomicSub(&deg[u], 1u);
                }
            }
            __syncthreads();
        }
        for (uint32_t i = a + tid; i < b; i += NT) gone += deg[order[i]];
        a = b;
        b = s_end;
        r++;
        __syncthreads();   // every thread has read s_end before it grows again
    }
    if (tid == 0) {
        PeelCtrl* c = P.ctrl;
        c->kmax = k;
        c->nlevels = nlev;
        c->rounds = r;
        c->grid_rounds = r;
        c->items = items;
        c->bytes = items * 4ull + n * 20ull;
    }
}

__global__ void k_peel_init(uint32_t n, const uint64_t* off, const uint64_t* split,
                            uint32_t* sl, uint32_t* alive0, uint64_t* wend, uint64_t* wnb,
                            PeelCtrl* c) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        sl[i] = kAlive;
        alive0[i] = (uint32_t)i;
        wend[i] = off[i + 1];
        wnb[i] = split ? split[i] : off[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->min_deg[0] = ~0ull;
        c->min_deg[1] = ~0ull;
    }
}

// Failure detection: the grid barrier of k_peel with one block withheld
// (absent >= 0), so that every other block's bounded wait runs out and sets
// the timeout flag; absent < 0 passes four barriers normally.
__global__ void k_barrier_probe(PeelCtrl* c, uint64_t wait_ns, int absent) {
    unsigned long long waited = 0;
    if ((int)blockIdx.x == absent) return;
    for (int i = 0; i < 4; i++)
        if (!grid_barrier(c, wait_ns, waited)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) c->barriers = 4;
}

template <int NT, int HC>
cudaError_t launch_peel(PeelParams& P, int sms, size_t smem, cudaStream_t s, unsigned* grid_out) {
    // opt in for every launch: the 48 KB default bounds static + dynamic
    // shared memory together, and the attribute persists across calls
    cudaError_t e = cudaFuncSetAttribute((k_peel<NT, HC>), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (k_peel<NT, HC>), NT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm <= 0) return cudaErrorInvalidConfiguration;
    // one block per SM: the fewest barrier arrivals
    unsigned grid = (unsigned)sms;
    *grid_out = grid;
    void* args[] = {&P};
    e = cudaLaunchCooperativeKernel((void*)k_peel<NT, HC>, dim3(grid), dim3(NT), args, smem, s);
    note_launch();
    return e;
}

dsd_status run_peel2_block(dsd_graph* g, uint32_t n, const uint64_t* off, const uint32_t* adj,
                           uint64_t mu0, uint64_t* core, uint32_t* rnd, uint64_t* lvl_k,
                           uint32_t* lvl_size, uint64_t* lvl_mu, PeelResult* res,
                           uint64_t kstart) {
    cudaStream_t s = g->stream;
    PeelCtrl* ctrl = nullptr;
    DSD_TRY(dalloc(&ctrl, 1, s));
    Peel2Block P{n, off, adj, core, rnd, lvl_k, lvl_size, lvl_mu, ctrl, mu0,
                 kstart ? (uint32_t)(kstart - 1) : 0u};
    const size_t smem = peel2_block_smem(n);
    PeelCtrl hc;
    cudaError_t e = cudaMemsetAsync(ctrl, 0, sizeof(PeelCtrl), s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_peel2_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)peel2_block_smem(kOneBlockN));
    if (e == cudaSuccess) {
        k_peel2_block<<<1, 1024, smem, s>>>(P);
        note_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, ctrl, sizeof(hc), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dev_free(ctrl, s);
    if (e != cudaSuccess) return cuda_fail(e, "h = 2 peel", __FILE__, __LINE__);
    res->kmax = hc.kmax;
    res->nlevels = hc.nlevels;
    res->rounds = hc.rounds;
    res->grid_rounds = hc.grid_rounds;
    res->items = hc.items;
    res->bytes = hc.bytes;
    res->threads = 1024;
    res->grid = 1;
    return DSD_OK;
}

}  // namespace

dsd_status run_peel(dsd_graph* g, int h, uint32_t n, const uint64_t* off, const uint32_t* adj,
                    const uint64_t* split, uint32_t maxdplus, unsigned long long* deg,
                    uint64_t mu0, uint64_t* core, uint32_t* rnd, uint64_t* lvl_k,
                    uint32_t* lvl_size, uint64_t* lvl_mu, PeelResult* res,
                    uint64_t kstart, uint64_t* snap) {
    cudaStream_t s = g->stream;
    *res = PeelResult();
    if (n == 0) return DSD_OK;
    if (h == 2 && n <= kOneBlockN && 2 * g->m <= kOneBlockAdj && !snap && kstart < (1u << 31))
        return run_peel2_block(g, n, off, adj, mu0, core, rnd, lvl_k, lvl_size, lvl_mu, res,
                               kstart);
    int sms = 152;
    DSD_TRY(num_sms(&sms));
    PeelParams P;
    memset(&P, 0, sizeof(P));
    P.n = n;
    P.h = h;
    P.off = off;
    P.deg = deg;
    P.core = core;
    P.rnd = rnd;
    P.lvl_k = lvl_k;
    P.lvl_size = lvl_size;
    P.lvl_mu = lvl_mu;
    P.wait_ns = wait_limit_ns();
    P.mu0 = mu0;
    P.k0 = kstart ? kstart - 1 : 0;
    P.snap = snap;
    P.cap = maxdplus < 32 ? 32 : maxdplus;
    P.warp_cand = warp_cand_limit(h);
    P.gather_cap = P.warp_cand;
    P.compact = h >= 3 ? 1 : 0;
    P.band_max = peel_tail_limit();
    // Big items (candidate sets above warp_cand vertices) for h >= 4; every
    // candidate set fits 32-word rows.
    const bool big_items = h >= 4;
    // Shared memory: per-warp candidate buffers (h >= 3), which share the
    // space of the bitmap search's (h >= 4)
    constexpr int NT = 1024;
    size_t work = h >= 3 ? (size_t)(NT / 32) * kWarpWords : 0;
    if (h >= 4) work = bitmap_words(kBitmapMax, NT / 32) + (h == 4 ? kBitmapMax / 2 : 0);
    // neighbourhood bitmaps for frontier vertices with the longest rows (a
    // binary search there takes 10 or more probes): up to 64 per round, two
    // sets, within 64 MiB
    if (h >= 3) {
        P.hub_words = ((uint64_t)n + 31) / 32;
        uint64_t slots = (64ull << 20) / (2 * 4 * P.hub_words);
        P.hub_slots = (uint32_t)(slots > 64 ? 64 : (slots < 4 ? 0 : slots));
    }
    const size_t smem = work * 4;

    uint32_t* sl = nullptr;
    uint32_t* lists = nullptr;
    uint64_t* wmeta = nullptr;
    uint32_t* wadj = nullptr;
    PeelCtrl* ctrl = nullptr;
    uint64_t* recs = nullptr;
    Band* bands = nullptr;
    uint2* big = nullptr;
    uint32_t* mid = nullptr;
    uint32_t* heavy = nullptr;
    uint32_t* xl = nullptr;
    uint32_t* hub_bm = nullptr;
    uint32_t* hubs = nullptr;
    uint32_t* blkcnt = nullptr;
    dsd_status st = DSD_OK;
    PeelCtrl hc;
    unsigned grid = 0;
    cudaError_t e = cudaSuccess;
    const uint64_t nadj = 2 * g->m;   // both CSRs of g hold 2m entries
    if ((st = dalloc(&sl, n, s)) != DSD_OK) goto done;
    if ((st = dalloc(&lists, (size_t)8 * n, s)) != DSD_OK) goto done;
    if ((st = dalloc(&blkcnt, (size_t)sms, s)) != DSD_OK) goto done;
    if ((st = dalloc(&wmeta, (size_t)2 * n, s)) != DSD_OK) goto done;
    if ((st = dalloc(&recs, (size_t)3 * n, s)) != DSD_OK) goto done;
    if ((st = dalloc(&wadj, nadj + 1, s)) != DSD_OK) goto done;
    if ((st = dalloc(&ctrl, 1, s)) != DSD_OK) goto done;
    if (P.band_max && (st = dalloc(&bands, kMaxBands, s)) != DSD_OK) goto done;
    if (big_items) {
        P.big_cap = g->m * 2 + 1;
        if ((st = dalloc(&big, P.big_cap, s)) != DSD_OK) goto done;
        // mid items (sets of warp_cand + 1 .. 32 candidates): up to 2^20 per
        // round (144 MB), the rest as big items
        uint64_t mc = P.big_cap < (1u << 20) ? P.big_cap : (1u << 20);
        if (mc > peel_item_mid_limit()) mc = peel_item_mid_limit();
        if (P.warp_cand < kWarpCand && mc > 0) {
            if ((st = dalloc(&mid, (size_t)mc * kMidWords, s)) != DSD_OK) goto done;
            P.mid = mid;
            P.mid_cap = (uint32_t)mc;
            P.gather_cap = kWarpCand;
        }
    }
    if (h >= 3 && (st = dalloc(&heavy, (size_t)2 * n, s)) != DSD_OK) goto done;
    P.heavy = heavy;
    P.vlist = heavy + n;
    if (big_items && P.cap > kBitmapMax &&
        (st = dalloc(&xl, (size_t)sms * (kMaxDepth + 1) * P.cap, s)) != DSD_OK)
        goto done;
    P.xl = xl;
    if (P.hub_slots) {
        if ((st = dalloc(&hub_bm, (size_t)2 * P.hub_slots * P.hub_words, s)) != DSD_OK) goto done;
        if ((st = dalloc(&hubs, (size_t)2 * P.hub_slots, s)) != DSD_OK) goto done;
        e = cudaMemsetAsync(hub_bm, 0, (size_t)2 * P.hub_slots * P.hub_words * 4, s);
        if (e != cudaSuccess) {
            st = cuda_fail(e, "peel bitmaps", __FILE__, __LINE__);
            goto done;
        }
    }
    P.hub_bm = hub_bm;
    P.hubs = hubs;
    P.sl = sl;
    P.alive[0] = lists;
    P.alive[1] = lists + n;
    P.front[0] = lists + 2 * (size_t)n;
    P.front[1] = lists + 3 * (size_t)n;
    P.front[2] = lists + 4 * (size_t)n;
    P.mem = lists + 5 * (size_t)n;
    P.band_of = lists + 6 * (size_t)n;
    P.t_size = lists + 7 * (size_t)n;
    P.blkcnt = blkcnt;
    P.c0 = reinterpret_cast<unsigned long long*>(recs);
    P.t_k = recs + n;
    P.t_mu = recs + 2 * (size_t)n;
    P.bands = bands;
    P.nadj = adj;
    P.nsplit = split ? split : off;
    P.wend = wmeta;
    P.wnb = wmeta + n;
    P.wadj = wadj;
    P.big = big;
    P.ctrl = ctrl;
    e = cudaMemsetAsync(ctrl, 0, sizeof(PeelCtrl), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(P.t_size, 0, (size_t)n * 4, s);
    if (e == cudaSuccess && nadj) e = cudaMemcpyAsync(wadj, adj, nadj * 4, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) {
        k_peel_init<<<sms * 4, 256, 0, s>>>(n, off, h >= 3 ? split : nullptr, sl, P.alive[0],
                                            P.wend, P.wnb, ctrl);
        note_launch();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = h == 2   ? launch_peel<NT, 2>(P, sms, smem, s, &grid)
            : h == 3 ? launch_peel<NT, 3>(P, sms, smem, s, &grid)
            : h == 4 ? launch_peel<NT, 4>(P, sms, smem, s, &grid)
                     : launch_peel<NT, 5>(P, sms, smem, s, &grid);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, ctrl, sizeof(PeelCtrl), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        st = cuda_fail(e, "peel", __FILE__, __LINE__);
        goto done;
    }
    if (hc.error & kErrTimeout) {
        set_error("a grid barrier wait in the peeling kernel exceeded %llu ms",
                  (unsigned long long)(P.wait_ns / 1000000ull));
        st = DSD_ERR_TIMEOUT;
        goto done;
    }
    if (hc.error) {
        set_error("peeling kernel internal error %u", hc.error);
        st = DSD_ERR_INTERNAL;
        goto done;
    }
    res->kmax = hc.kmax;
    res->nlevels = hc.nlevels;
    res->rounds = hc.rounds;
    res->items = hc.items;
    res->bytes = hc.bytes;
    res->barrier_ns = hc.barrier_ns;
    res->barriers = hc.barriers;
    res->compactions = hc.compactions;
    res->threads = NT;
    res->grid = grid;
    res->grid_rounds = hc.grid_rounds;
    res->band_n = hc.band_n;
    res->band_round = hc.band_round;
    res->bands = hc.nbands;
    res->phase2_ns = hc.phase2_ns;
    for (int i = 0; i < 8; i++) res->tph[i] = hc.tph[i];
done:
    dev_free(sl, s);
    dev_free(lists, s);
    dev_free(wmeta, s);
    dev_free(wadj, s);
    dev_free(ctrl, s);
    dev_free(recs, s);
    dev_free(bands, s);
    dev_free(big, s);
    dev_free(mid, s);
    dev_free(heavy, s);
    dev_free(xl, s);
    dev_free(hub_bm, s);
    dev_free(hubs, s);
    dev_free(blkcnt, s);
    return st;
}

}  // namespace dsd

extern "C" dsd_status dsd_check_barrier_timeout(int absent_block, uint32_t wait_ms,
                                                void* cuda_stream) {
    using namespace dsd;
    set_error("");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int sms = 152;
    DSD_TRY(num_sms(&sms));
    if (wait_ms == 0 || wait_ms > 60000 || absent_block >= sms) {
        set_error("dsd_check_barrier_timeout: need 0 < wait_ms <= 60000 and absent_block < %d",
                  sms);
        return DSD_ERR_INVALID;
    }
    PeelCtrl* ctrl = nullptr;
    DSD_TRY(dalloc(&ctrl, 1, s));
    PeelCtrl hc;
    memset(&hc, 0, sizeof(hc));
    uint64_t wait_ns = (uint64_t)wait_ms * 1000000ull;
    int absent = absent_block;
    void* args[] = {&ctrl, &wait_ns, &absent};
    cudaError_t e = cudaMemsetAsync(ctrl, 0, sizeof(PeelCtrl), s);
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel((void*)k_barrier_probe, dim3(sms), dim3(128), args, 0, s);
    note_launch();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, ctrl, sizeof(hc), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dev_free(ctrl, s);
    if (e != cudaSuccess) return cuda_fail(e, "barrier probe", __FILE__, __LINE__);
    if (hc.error & kErrTimeout) {
        set_error("grid barrier wait ran out after %u ms (block %d withheld)", wait_ms, absent);
        return DSD_ERR_TIMEOUT;
    }
    if (hc.error || hc.barriers != 4) {
        set_error("barrier probe: error %u, %u barriers", hc.error, hc.barriers);
        return DSD_ERR_INTERNAL;
    }
    return DSD_OK;
}
