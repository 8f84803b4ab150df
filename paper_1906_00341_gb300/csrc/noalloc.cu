// Allocation-free triangle clique-degrees (h = 3) for callers that cannot
// allocate device memory.
//
// Some callers cannot call cudaMalloc: plug-ins that live inside a host
// framework whose allocator has already reserved the device memory (another
// allocation would fail or fragment the framework's pool), and latency-bound
// serving paths where an allocation's cost or possible failure in the middle
// of a request is not acceptable.  dsd_triangle_degrees_noalloc serves them:
// it reads the caller's CSR, writes the caller's output buffers, and keeps
// its own scratch (work counters and lists of longer rows) in one statically
// sized __device__ array of this translation unit.  It calls no allocator.
//
// The first call on a device looks up the array's device address (with that
// device current) and caches it; make that first call before any stream
// capture begins.
//
// Unlike dsd_clique_degrees it needs no graph handle and no degeneracy
// order: rows are oriented by vertex id (N+(u) = the entries of row u that
// exceed u), which lists every triangle exactly once, like any total order.
//
// The scratch array is shared by every call in the process on that device:
// calls whose work overlaps on the GPU (different streams, or different host
// threads) race on it.  Serialise them.
#include "common.cuh"

#include <mutex>

namespace dsd {
namespace {

// Scratch: [0] light rows taken, [1] medium rows, [2] large rows, [3] and [4]
// those taken; from word kListAt on the medium rows, from the end down the
// large ones (together at most n).
constexpr uint32_t kListAt = 8;
constexpr uint32_t kNoAllocWords = 1u << 20;           // 4 MiB
constexpr uint32_t kNoAllocMaxN = kNoAllocWords - 64;  // every row fits the list
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocWords];

constexpr int kDevMax = 64;
uint32_t* g_scratch_ptr[kDevMax];
std::once_flag g_scratch_once[kDevMax];
cudaError_t g_scratch_err[kDevMax];

__device__ __forceinline__ uint64_t tail_start(const uint64_t* off, const uint32_t* adj,
                                               uint32_t u) {
    uint64_t b = off[u], e = off[u + 1];
    return b + lower_bound_u32(adj + b, e - b, u + 1u);
}

// A row's tail (entries above its own id) has d entries: light up to 32,
// medium up to kMediumMax, large above.  Every entry y of N+(x), x in N+(u), is
// looked up among N+(u): by binary search in a warp's 32 entries, else in a
// hash table in shared memory whose slots hold an id and its count, so that a
// look-up is one or two shared loads instead of a binary search through the
// row (10-14 dependent loads in L2) and a triangle no global atomic.  Where
// N+(x) begins is searched for by a lane an x, all at once; one after another
// each search was a chain of dependent global loads.  Bound by the look-ups
// (shared loads) and by the row loads from L2.  777,777 vertices of a power
// law, 7.8M draws, hubs first: 37.5 -> 8.8 ms.
constexpr uint32_t kMediumMax = 1024;
constexpr uint32_t kMediumSlots = 2048;
constexpr uint32_t kLargeMax = 12288;    // larger rows keep the table-free path
constexpr uint32_t kLargeSlots = 16384;

// Light rows: one warp each (dynamic queue).  The others are listed.
__global__ void __launch_bounds__(256) k_na_light(uint32_t n, const uint64_t* off,
                                                  const uint32_t* adj,
                                                  unsigned long long* deg,
                                                  unsigned long long* mu, uint32_t* scratch) {
    __shared__ uint32_t sC[8][32];
    __shared__ unsigned sCnt[8][32];
    unsigned lane = lane_id(), w = warp_id();
    uint32_t* C = sC[w];
    unsigned* cnt = sCnt[w];
    unsigned long long acc = 0;
    for (;;) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(&scratch[0], 32u);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= n) break;
        // a lane a row: where its tail begins
        const uint32_t mine = base + lane;
        uint64_t tb = 0, te = 0;
        if (mine < n) {
            te = off[mine + 1];
            tb = tail_start(off, adj, mine);
        }
        const uint32_t md = (uint32_t)(te - tb);
        if (md > 32) {
            if (md <= kMediumMax) scratch[kListAt + atomicAdd(&scratch[1], 1u)] = mine;
            else scratch[kNoAllocWords - 1 - atomicAdd(&scratch[2], 1u)] = mine;
        }
        unsigned todo = __ballot_sync(0xffffffffu, md >= 2 && md <= 32);
        while (todo) {
            const int q = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t u = base + q;
            const uint64_t b = __shfl_sync(0xffffffffu, tb, q);
            const uint32_t d = __shfl_sync(0xffffffffu, md, q);
            uint32_t x = 0;
            uint64_t xb = 0, xe = 0;
            if (lane < d) {
                x = adj[b + lane];
                C[lane] = x;
                cnt[lane] = 0;
                xe = off[x + 1];
                xb = tail_start(off, adj, x);
            }
            __syncwarp();
            const uint32_t cmax = C[d - 1];
            unsigned long long t = 0;
            for (uint32_t i = 0; i + 1 < d; i++) {
                const uint64_t rb = __shfl_sync(0xffffffffu, xb, i);
                const uint64_t re = __shfl_sync(0xffffffffu, xe, i);
                unsigned hits = 0;
                for (uint64_t p0 = rb; p0 < re; p0 += 32) {
                    const uint64_t p = p0 + lane;
                    const uint32_t y = p < re ? adj[p] : kNone;
                    if (y <= cmax) {
                        uint32_t pos = (uint32_t)lower_bound_u32(C, d, y);
                        if (pos < d && C[pos] == y) { atomicAdd(&cnt[pos], 1u); hits++; }
                    }
                    if (__shfl_sync(0xffffffffu, y, 31) > cmax) break;
                }
                hits = __reduce_add_sync(0xffffffffu, hits);
                if (lane == 0 && hits) atomicAdd(&cnt[i], hits);
                t += hits;
            }
            __syncwarp();
            if (t) {
                if (lane < d && cnt[lane]) atomicAdd(&deg[C[lane]], (unsigned long long)cnt[lane]);
                if (lane == 0) { atomicAdd(&deg[u], t); acc += t; }
            }
            __syncwarp();
        }
    }
    if (lane == 0 && acc) atomicAdd(mu, acc);
}

// Medium (LARGE = false) and large rows: a block each, taken from the list.
// Dynamic shared memory: ids and counts of SLOTS slots, then where each
// candidate's tail begins and ends (MAXD entries of offset and length).
template <int NT, uint32_t SLOTS, uint32_t MAXD, bool LARGE>
__global__ void __launch_bounds__(NT) k_na_hash(const uint64_t* off, const uint32_t* adj,
                                                unsigned long long* deg, unsigned long long* mu,
                                                uint32_t* scratch) {
    extern __shared__ __align__(16) uint32_t sm[];
    uint32_t* key = sm;
    uint32_t* cnt = key + SLOTS;
    uint32_t* rel = cnt + SLOTS;      // tail start within the candidate's row
    __shared__ unsigned long long s_tot;
    __shared__ uint32_t s_it;
    const unsigned lane = lane_id(), wid = warp_id(), nw = NT / 32;
    const uint32_t rows = scratch[LARGE ? 2 : 1];
    for (;;) {
        if (threadIdx.x == 0) {
            s_it = atomicAdd(&scratch[LARGE ? 4 : 3], 1u);
            s_tot = 0;
        }
        __syncthreads();
        const uint32_t it = s_it;
        if (it >= rows) break;
        const uint32_t u = LARGE ? scratch[kNoAllocWords - 1 - it] : scratch[kListAt + it];
        const uint64_t b = tail_start(off, adj, u), e = off[u + 1];
        const uint32_t d = (uint32_t)(e - b);
        const uint32_t* C = adj + b;
        const uint32_t cmax = C[d - 1];
        const bool table = d <= MAXD;
        uint32_t slots = 64;
        while (slots < 2 * d && slots < SLOTS) slots <<= 1;
        const uint32_t mask = slots - 1, shift = 32u - (uint32_t)__popc(mask);
        if (table) {
            for (uint32_t i = threadIdx.x; i < slots; i += NT) {
                key[i] = kNone;
                cnt[i] = 0;
            }
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < d; i += NT) {
                const uint32_t x = C[i];
                uint32_t s = (x * 2654435761u) >> shift;
                while (atomicCAS(&key[s], kNone, x) != kNone) s = (s + 1) & mask;
                rel[i] = (uint32_t)(tail_start(off, adj, x) - off[x]);
            }
        }
        __syncthreads();
        unsigned long long mine = 0;
        for (uint32_t i = wid; i < d; i += nw) {
            const uint32_t x = C[i];
            const uint64_t xe = off[x + 1];
            const uint64_t xb = table ? off[x] + rel[i] : tail_start(off, adj, x);
            unsigned hits = 0;
            for (uint64_t p0 = xb; p0 < xe; p0 += 128) {
                uint32_t ys[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint64_t p = p0 + 32 * q + lane;
                    ys[q] = p < xe ? adj[p] : kNone;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t y = ys[q];
                    if (y > cmax) continue;
                    if (table) {
                        uint32_t s = (y * 2654435761u) >> shift, k = key[s];
                        while (k != y && k != kNone) {
                            s = (s + 1) & mask;
                            k = key[s];
                        }
                        if (k == y) {
                            atomicAdd(&cnt[s], 1u);
                            hits++;
                        }
                    } else {
                        const uint64_t pos = lower_bound_u32(C, d, y);
                        if (pos < d && C[pos] == y) {
                            atomicAdd(&deg[y], 1ull);
                            hits++;
                        }
                    }
                }
                if (__shfl_sync(0xffffffffu, ys[3], 31) > cmax) break;
            }
            hits = __reduce_add_sync(0xffffffffu, hits);
            if (lane == 0 && hits) {
                if (table) {
                    uint32_t s = (x * 2654435761u) >> shift;
                    while (key[s] != x) s = (s + 1) & mask;
                    atomicAdd(&cnt[s], hits);
                } else {
                    atomicAdd(&deg[x], (unsigned long long)hits);
                }
                mine += hits;
            }
        }
        if (mine) atomicAdd(&s_tot, mine);
        __syncthreads();
        if (table)
            for (uint32_t i = threadIdx.x; i < slots; i += NT)
                if (cnt[i] && key[i] != kNone) atomicAdd(&deg[key[i]], (unsigned long long)cnt[i]);
        if (threadIdx.x == 0 && s_tot) {
            atomicAdd(&deg[u], s_tot);
            atomicAdd(mu, s_tot);
        }
        __syncthreads();
    }
}

constexpr size_t kMediumBytes = (2 * kMediumSlots + kMediumMax) * sizeof(uint32_t);
constexpr size_t kLargeBytes = (2 * kLargeSlots + kLargeMax) * sizeof(uint32_t);
constexpr auto* kLarge = k_na_hash<1024, kLargeSlots, kLargeMax, true>;

// Device address of the scratch array for the current device, looked up
// once per device (with that device current).
dsd_status scratch_for_current_device(uint32_t** out) {
    int dev = 0;
    DSD_CU(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kDevMax) {
        set_error("device ordinal %d out of range", dev);
        return DSD_ERR_UNSUPPORTED;
    }
    std::call_once(g_scratch_once[dev], [dev]() {
        void* p = nullptr;
        g_scratch_err[dev] = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        g_scratch_ptr[dev] = static_cast<uint32_t*>(p);
        if (g_scratch_err[dev] == cudaSuccess)   // once: later calls may run under capture
            g_scratch_err[dev] = cudaFuncSetAttribute(
                kLarge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLargeBytes);
    });
    if (g_scratch_err[dev] != cudaSuccess || !g_scratch_ptr[dev]) {
        set_error("look-up of the scratch array failed: %s",
                  cudaGetErrorString(g_scratch_err[dev]));
        return DSD_ERR_CUDA;
    }
    *out = g_scratch_ptr[dev];
    return DSD_OK;
}

}  // namespace
}  // namespace dsd

using namespace dsd;

extern "C" dsd_status dsd_triangle_degrees_noalloc(uint32_t n, const uint64_t* off,
                                                   const uint32_t* adj, uint64_t* deg,
                                                   uint64_t* mu, void* cuda_stream) {
    set_error("");
    if (!off || !deg || !mu) {
        set_error("dsd_triangle_degrees_noalloc: off, deg and mu must be device pointers");
        return DSD_ERR_INVALID;
    }
    if (n > kNoAllocMaxN) {
        set_error("dsd_triangle_degrees_noalloc handles at most %u vertices (got %u): its "
                  "scratch is a fixed %u-word device array", kNoAllocMaxN, n, kNoAllocWords);
        return DSD_ERR_UNSUPPORTED;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (n && !adj) {
        // an edgeless CSR may come with a null adj (a zero-length device
        // buffer has no address); any other null adj is an error
        uint64_t edges = 0;
        DSD_CU(cudaMemcpyAsync(&edges, off + n, sizeof(edges), cudaMemcpyDeviceToHost, s));
        DSD_CU(cudaStreamSynchronize(s));
        if (edges) {
            set_error("dsd_triangle_degrees_noalloc: adj is NULL but off[n] = %llu",
                      (unsigned long long)edges);
            return DSD_ERR_INVALID;
        }
    }
    uint32_t* scratch = nullptr;
    DSD_TRY(scratch_for_current_device(&scratch));
    // the counters and the outputs start at zero on every call
    DSD_CU(cudaMemsetAsync(scratch, 0, kListAt * sizeof(uint32_t), s));
    DSD_CU(cudaMemsetAsync(deg, 0, (size_t)n * sizeof(uint64_t), s));
    DSD_CU(cudaMemsetAsync(mu, 0, sizeof(uint64_t), s));
    if (n == 0) return DSD_OK;
    int sms = 152;
    DSD_TRY(num_sms(&sms));
    k_na_light<<<sms * 8, 256, 0, s>>>(n, off, adj, (unsigned long long*)deg,
                                       (unsigned long long*)mu, scratch);
    note_launch();
    // in one stream: the medium rows wait for the last large one
    kLarge<<<sms, 1024, kLargeBytes, s>>>(off, adj, (unsigned long long*)deg,
                                          (unsigned long long*)mu, scratch);
    note_launch();
    k_na_hash<256, kMediumSlots, kMediumMax, false><<<sms * 8, 256, kMediumBytes, s>>>(
        off, adj, (unsigned long long*)deg, (unsigned long long*)mu, scratch);
    note_launch();
    DSD_CU(cudaGetLastError());
    return DSD_OK;
}
