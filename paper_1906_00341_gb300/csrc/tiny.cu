// CSR build and orientation of small graphs by one block.
//
// A graph of a few thousand vertices is launch-bound: the general builders
// take some 20 launches each (scans, a sort per row class, copies) with a few
// microseconds of work in all.  Here one block does a whole stage with its
// counters in shared memory: G(2000, 0.005), edge list to outputs, 0.93 ->
// 0.82 ms.  Bound by the latency of the row sorts and of the passes over the
// edge list, one SM's worth; the limits below are where the general path's
// launches cost about as much.
#include "graph.cuh"
#include "tiny.cuh"

namespace dsd {
namespace {

constexpr int NT = 1024, NW = NT / 32;
constexpr uint32_t kWarpRow = 256;              // a warp's sort buffer
constexpr uint32_t kBlockRow = NW * kWarpRow;   // 8192: all of them together
static_assert(kBlockRow >= kTinyN, "a row without repeats fits the block's buffer");

// Rows above kWarpRow are sorted one after another by the whole block, each
// some 2 (4 + N / 128) us, padded to N entries (50 rows of 300 entries: the
// CSR 0.49 ms, 0.21 by the general path; 20 of 1,600: 0.41 and 0.23; 4 of
// 2,900: 0.28 and 0.39 before its pool): above this sum of 4 + N / 128 the
// general path sorts them side by side.
constexpr uint32_t kLongBudget = 192;

struct TinyOut {
    unsigned long long total;   // entries of the cleaned CSR
    uint32_t err;               // an endpoint out of range
    uint32_t big;               // rows (with repeats) too long, or too many long ones
    uint32_t dmax;              // largest |N+(v)|
};

// Exclusive prefix sums of a[0..n) in place (shared memory); a[n] = the total.
__device__ uint32_t prefix(uint32_t* a, uint32_t n, uint32_t* s_w) {
    const unsigned lane = lane_id(), wid = warp_id();
    uint32_t run = 0;
    for (uint32_t t0 = 0; t0 < n; t0 += NT) {
        const uint32_t i = t0 + threadIdx.x, v = i < n ? a[i] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if ((int)lane >= o) x += y;
        }
        if (lane == 31) s_w[wid] = x;
        __syncthreads();
        uint32_t w = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if ((int)lane >= o) w += y;
        }
        const uint32_t before = wid ? __shfl_sync(0xffffffffu, w, wid - 1) : 0u;
        const uint32_t all = __shfl_sync(0xffffffffu, w, 31);
        if (i < n) a[i] = run + before + x - v;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) a[n] = run;
    __syncthreads();
    return run;
}

// Bitonic network over s[0..N) by threads `t` of `nt`, `sync` between steps.
template <class Sync>
__device__ __forceinline__ void bitonic(uint32_t* s, uint32_t N, uint32_t t, uint32_t nt,
                                        Sync sync) {
    for (uint32_t k = 2; k <= N; k <<= 1)
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t x = t; x < N; x += nt) {
                const uint32_t y = x ^ j;
                if (y > x) {
                    const bool asc = (x & k) == 0;
                    const uint32_t a = s[x], b = s[y];
                    if ((a > b) == asc) {
                        s[x] = b;
                        s[y] = a;
                    }
                }
            }
            sync();
        }
}

// The unique entries of sorted s[0..l) to row, one warp; their number.
__device__ __forceinline__ uint32_t write_unique(const uint32_t* s, uint32_t l, uint32_t* row) {
    const unsigned lane = lane_id();
    uint32_t out = 0;
    for (uint32_t b0 = 0; b0 < l; b0 += 32) {
        const uint32_t x = b0 + lane;
        const uint32_t v = x < l ? s[x] : 0u;
        const bool keep = x < l && (x == 0 || v != s[x - 1]);
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (keep) row[out + __popc(bal & ((1u << lane) - 1u))] = v;
        out += __popc(bal);
    }
    return out;
}

// Sorts row v = vals[pos[v] .. pos[v] + len[v]) for every v in place and drops
// repeats; len[v] becomes the unique length.  A warp a row (in registers up
// to 32 entries), rows above kWarpRow by the block.  buf: kBlockRow words.
__device__ void sort_rows(uint32_t* vals, const uint32_t* pos, uint32_t* len, uint32_t n,
                          uint32_t* buf, uint32_t* longs, uint32_t* s_nl) {
    const unsigned lane = lane_id(), wid = warp_id();
    if (threadIdx.x == 0) *s_nl = 0;
    __syncthreads();
    uint32_t* sw = buf + wid * kWarpRow;
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
            __syncwarp();
            if (lane == 0) len[v] = __popc(b);
        } else if (l <= kWarpRow) {
            uint32_t N = 64;
            while (N < l) N <<= 1;
            for (uint32_t j = lane; j < N; j += 32) sw[j] = j < l ? row[j] : kNone;
            __syncwarp();
            bitonic(sw, N, lane, 32, [] { __syncwarp(); });
            const uint32_t u = write_unique(sw, l, row);
            __syncwarp();
            if (lane == 0) len[v] = u;
        } else if (lane == 0) {
            longs[atomicAdd(s_nl, 1u)] = v;
        }
    }
    __syncthreads();
    const uint32_t nl = *s_nl;
    for (uint32_t i = 0; i < nl; i++) {
        const uint32_t v = longs[i], l = len[v];
        uint32_t* row = vals + pos[v];
        uint32_t N = 512;
        while (N < l) N <<= 1;
        for (uint32_t j = threadIdx.x; j < N; j += NT) buf[j] = j < l ? row[j] : kNone;
        __syncthreads();
        bitonic(buf, N, threadIdx.x, NT, [] { __syncthreads(); });
        if (wid == 0) {
            const uint32_t u = write_unique(buf, l, row);
            if (lane == 0) len[v] = u;
        }
        __syncthreads();
    }
}

// Shared words: two arrays of n + 1, the sort buffer, the list of long rows
// (a row above kWarpRow has more than that many of the entries).
constexpr uint32_t kLongs = 2 * kTinyM / kWarpRow + 1;
constexpr size_t tiny_words(uint32_t n) { return 2 * ((size_t)n + 1) + kBlockRow + kLongs; }

// Edge list -> cleaned CSR.  tmp: 2m entries; adj: room for 2m.
__global__ void __launch_bounds__(NT, 1) k_tiny_csr(uint32_t n, uint32_t m, const uint32_t* src,
                                                    const uint32_t* dst, uint32_t* tmp,
                                                    uint64_t* off, uint32_t* adj, TinyOut* out) {
    extern __shared__ uint32_t sm[];
    uint32_t* pos = sm;
    uint32_t* len = pos + n + 1;
    uint32_t* buf = len + n + 1;
    uint32_t* longs = buf + kBlockRow;
    __shared__ uint32_t s_w[32], s_nl, s_err, s_big;
    const unsigned lane = lane_id(), wid = warp_id();
    for (uint32_t v = threadIdx.x; v <= n; v += NT) pos[v] = len[v] = 0;
    if (threadIdx.x == 0) s_err = s_big = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < m; i += NT) {
        const uint32_t u = src[i], v = dst[i];
        if (u >= n || v >= n) {
            s_err = 1;
            continue;
        }
        if (u == v) continue;
        atomicAdd(&pos[u], 1u);
        atomicAdd(&pos[v], 1u);
    }
    __syncthreads();
    for (uint32_t v = threadIdx.x; v < n; v += NT) {
        const uint32_t l = pos[v];
        if (l <= kWarpRow) continue;
        uint32_t N = 512;
        while (N < l) N <<= 1;
        atomicAdd(&s_big, l > kBlockRow ? kLongBudget + 1u : 4u + N / 128u);
    }
    __syncthreads();
    if (s_err || s_big > kLongBudget) {
        if (threadIdx.x == 0) *out = TinyOut{0, s_err, 1, 0};
        return;
    }
    (void)prefix(pos, n, s_w);
    for (uint32_t i = threadIdx.x; i < m; i += NT) {
        const uint32_t u = src[i], v = dst[i];
        if (u == v) continue;
        tmp[pos[u] + atomicAdd(&len[u], 1u)] = v;
        tmp[pos[v] + atomicAdd(&len[v], 1u)] = u;
    }
    __syncthreads();
    sort_rows(tmp, pos, len, n, buf, longs, &s_nl);
    const uint32_t total = prefix(len, n, s_w);   // row starts of the cleaned CSR
    for (uint32_t v = threadIdx.x; v <= n; v += NT) off[v] = len[v];
    for (uint32_t v = wid; v < n; v += NW) {
        const uint32_t from = pos[v], to = len[v], l = len[v + 1] - to;
        for (uint32_t j = lane; j < l; j += 32) adj[to + j] = tmp[from + j];
    }
    if (threadIdx.x == 0) *out = TinyOut{total, 0, 0, 0};
}

// Rank by (round, id), relabelled sorted rows, N+ starts.
__global__ void __launch_bounds__(NT, 1) k_tiny_orient(uint32_t n, const uint64_t* off,
                                                       const uint32_t* adj, const uint32_t* rnd,
                                                       uint32_t* new_of, uint32_t* old_of,
                                                       uint64_t* roff, uint32_t* radj,
                                                       uint64_t* split, TinyOut* out) {
    extern __shared__ uint32_t sm[];
    uint32_t* rank = sm;            // caller id -> rank
    uint32_t* pos = rank + n + 1;   // by rank: length, then row start
    uint32_t* buf = pos + n + 1;
    uint32_t* longs = buf + kBlockRow;
    __shared__ uint32_t s_w[32], s_nl, s_dmax;
    const unsigned lane = lane_id(), wid = warp_id();
    uint32_t N = 32;
    while (N < n) N <<= 1;
    // rounds and ids stay below 2^16
    for (uint32_t v = threadIdx.x; v < N; v += NT) buf[v] = v < n ? (rnd[v] << 16) | v : kNone;
    if (threadIdx.x == 0) s_dmax = 0;
    __syncthreads();
    bitonic(buf, N, threadIdx.x, NT, [] { __syncthreads(); });
    for (uint32_t p = threadIdx.x; p < n; p += NT) {
        const uint32_t o = buf[p] & 0xffffu;
        rank[o] = p;
        old_of[p] = o;
        new_of[o] = p;
        pos[p] = (uint32_t)(off[o + 1] - off[o]);
    }
    __syncthreads();
    (void)prefix(pos, n, s_w);
    for (uint32_t p = threadIdx.x; p <= n; p += NT) roff[p] = pos[p];
    __syncthreads();
    for (uint32_t o = wid; o < n; o += NW) {
        const uint64_t from = off[o];
        const uint32_t to = pos[rank[o]], l = (uint32_t)(off[o + 1] - from);
        for (uint32_t j = lane; j < l; j += 32) radj[to + j] = rank[adj[from + j]];
    }
    __syncthreads();
    // the ranks are not needed any more: their array takes the lengths
    for (uint32_t p = threadIdx.x; p < n; p += NT) rank[p] = pos[p + 1] - pos[p];
    __syncthreads();
    sort_rows(radj, pos, rank, n, buf, longs, &s_nl);
    for (uint32_t p = threadIdx.x; p < n; p += NT) {
        const uint32_t b = pos[p], e = pos[p + 1];
        const uint32_t at = b + (uint32_t)lower_bound_u32(radj + b, e - b, p + 1u);
        split[p] = at;
        if (e > at) atomicMax(&s_dmax, e - at);
    }
    __syncthreads();
    if (threadIdx.x == 0) *out = TinyOut{pos[n], 0, 0, s_dmax};
}

dsd_status opt_in(const void* fn) {
    DSD_CU(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(tiny_words(kTinyN) * 4)));
    return DSD_OK;
}

}  // namespace

dsd_status tiny_csr(dsd_graph* g, uint32_t m, const uint32_t* src, const uint32_t* dst,
                    bool* done) {
    cudaStream_t s = g->stream;
    const uint32_t n = g->n;
    *done = false;
    DSD_TRY(opt_in((const void*)k_tiny_csr));
    uint32_t* tmp = nullptr;
    TinyOut* out = nullptr;
    uint64_t* off = nullptr;
    uint32_t* adj = nullptr;
    TinyOut h;
    dsd_status st = dalloc(&off, (size_t)n + 1, s);
    if (st == DSD_OK) st = dalloc(&adj, (size_t)2 * m + 1, s);
    if (st == DSD_OK) st = dalloc(&tmp, (size_t)2 * m + 16, s);
    if (st == DSD_OK) st = dalloc(&out, 1, s);
    if (st == DSD_OK) {
        k_tiny_csr<<<1, NT, tiny_words(n) * 4, s>>>(n, m, src, dst, tmp, off, adj, out);
        note_launch();
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, out, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_fail(e, "small CSR", __FILE__, __LINE__);
    }
    dev_free(tmp, s);
    dev_free(out, s);
    if (st == DSD_OK && h.err) {
        set_error("edge endpoint out of range (n = %u)", n);
        st = DSD_ERR_INVALID;
    }
    if (st != DSD_OK || h.big) {
        dev_free(off, s);
        dev_free(adj, s);
        return st;
    }
    g->off = off;
    g->adj = adj;
    g->m = h.total / 2;
    *done = true;
    return DSD_OK;
}

dsd_status tiny_orient(dsd_graph* g) {
    cudaStream_t s = g->stream;
    DSD_TRY(opt_in((const void*)k_tiny_orient));
    TinyOut* out = nullptr;
    TinyOut h;
    DSD_TRY(dalloc(&out, 1, s));
    k_tiny_orient<<<1, NT, tiny_words(g->n) * 4, s>>>(g->n, g->off, g->adj, g->rnd, g->new_of,
                                                      g->old_of, g->roff, g->radj, g->rsplit, out);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, out, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    dev_free(out, s);
    if (e != cudaSuccess) return cuda_fail(e, "small orientation", __FILE__, __LINE__);
    g->maxdplus = h.dmax;
    return DSD_OK;
}

}  // namespace dsd
