// Graph upload: device-side validation of the CSR (the paper's graphs are
// symmetric with positive integer weights: Table "preliminaries_notation",
// Section "Evaluation") and interleaving of (neighbour, weight) into one
// 8-byte record per arc, so a relaxation reads one sector-aligned pair.
#include <algorithm>
#include <atomic>

#include "internal.h"

namespace stn {

int current_sm_count() {
    constexpr int MAX_DEVICES = 64;
    static std::atomic<int> cache[MAX_DEVICES];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
        cudaGetLastError();
        dev = -1;
    }
    int sms = dev >= 0 ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (sms > 0) return sms;
    if (dev < 0 || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        sms < 1) {
        cudaGetLastError();
        return 1;
    }
    cache[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

enum : uint32_t {
    BAD_RANGE = 1u,      // neighbour id out of range
    BAD_SELF = 2u,       // self-loop
    BAD_WEIGHT = 4u,     // weight 0
    BAD_ORDER = 8u,      // row not strictly ascending (unsorted or duplicate)
    BAD_SYMMETRY = 16u,  // reverse arc missing or with another weight
};

__device__ __forceinline__ bool find_reverse(const uint32_t *row_ptr, const int32_t *col,
                                             const uint32_t *w, uint32_t v, uint32_t u,
                                             uint32_t wt) {
    uint32_t lo = row_ptr[v], hi = row_ptr[v + 1];
    while (lo < hi) {
        uint32_t mid = lo + (hi - lo) / 2;
        uint32_t c = (uint32_t)col[mid];
        if (c == u) return w[mid] == wt;
        if (c < u) lo = mid + 1; else hi = mid;
    }
    return false;
}

__global__ void __launch_bounds__(256) validate_kernel(const uint32_t *__restrict__ row_ptr,
                                                       const int32_t *__restrict__ col,
                                                       const uint32_t *__restrict__ w,
                                                       uint32_t n, uint2 *__restrict__ adj,
                                                       const uint32_t *__restrict__ new_of,
                                                       const uint32_t *__restrict__ new_row_ptr,
                                                       uint32_t *bad, uint32_t *max_w) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    uint32_t flags = 0, wmax = 0;
    for (uint32_t b0 = warp * 32; b0 < n; b0 += nwarps * 32) {
        uint32_t u = b0 + lane;
        uint32_t s = 0, deg = 0;
        if (u < n) {
            s = row_ptr[u];
            deg = row_ptr[u + 1] - s;
        }
        uint32_t incl = warp_inclusive_scan(deg);
        uint32_t excl = incl - deg;
        uint32_t total = __shfl_sync(FULL, incl, 31);
        for (uint32_t b = 0; b < total; b += 32) {
            uint32_t j = b + lane;
            bool valid = j < total;
            uint32_t owner = warp_owner_search(excl, valid ? j : 0);
            uint32_t so = __shfl_sync(FULL, s, owner);
            uint32_t eo = __shfl_sync(FULL, excl, owner);
            if (!valid) continue;
            uint32_t src = b0 + owner;
            uint32_t e = so + (j - eo);
            int32_t c = col[e];
            uint32_t wt = w[e];
            wmax = max(wmax, wt);
            if (c < 0 || (uint32_t)c >= n) {
                flags |= BAD_RANGE;
                continue;
            }
            if (new_of)
                adj[new_row_ptr[new_of[src]] + (e - so)] = make_uint2(new_of[c], wt);
            else
                adj[e] = make_uint2((uint32_t)c, wt);
            if ((uint32_t)c == src) flags |= BAD_SELF;
            if (wt == 0) flags |= BAD_WEIGHT;
            if (e > so && col[e - 1] >= c) flags |= BAD_ORDER;
            if (!find_reverse(row_ptr, col, w, (uint32_t)c, src, wt)) flags |= BAD_SYMMETRY;
        }
    }
    if (flags) atomicOr(bad, flags);
    wmax = __reduce_max_sync(FULL, wmax);
    if (lane == 0 && wmax) atomicMax(max_w, wmax);
}

// Rows split by weight: arcs lighter than delta first, then the rest, each
// part in the row's order.  Short rows go 32 to a warp, the consecutive rows'
// arcs read as one run: a lane counts its row's light arcs from the window's
// ballot, then every arc finds its place from its row's running count.  Hub
// rows take a block each.  (With a warp per row the longest hub held up the
// pass: R-MAT 26, degree 8, 19.7 ms against 3.2 + 3.6.)
constexpr uint32_t PART_HUB_DEG = 1024;
__global__ void __launch_bounds__(256) partition_kernel(const uint32_t *__restrict__ row_ptr,
                                                        const uint2 *__restrict__ adj, uint32_t n,
                                                        uint32_t delta, uint2 *__restrict__ adj_w,
                                                        uint32_t *__restrict__ lend) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t v0 = warp * 32; v0 < n; v0 += nwarps * 32) {
        const uint32_t v = v0 + lane;
        uint32_t s = 0, deg = 0;
        if (v < n) {
            s = row_ptr[v];
            deg = row_ptr[v + 1] - s;
        }
        const bool hub = deg >= PART_HUB_DEG;
        if (hub) deg = 0;
        const uint32_t incl = warp_inclusive_scan(deg), excl = incl - deg;
        const uint32_t total = __shfl_sync(FULL, incl, 31);
        // the lane's row inside the window [b, b + 32)
        auto window = [&](uint32_t b) {
            if (deg == 0 || excl >= b + 32 || incl <= b) return 0u;
            const uint32_t lo = excl > b ? excl - b : 0u, hi = min(incl - b, 32u);
            return (FULL >> (32 - (hi - lo))) << lo;
        };
        uint32_t nl = 0;
        for (uint32_t b = 0; b < total; b += 32) {
            const uint32_t j = b + lane;
            const uint32_t own = warp_owner_search(excl, j < total ? j : 0);
            const uint32_t at = __shfl_sync(FULL, s - excl, own) + j;
            const uint32_t ml = __ballot_sync(FULL, j < total && __ldg(&adj[at].y) < delta);
            nl += (uint32_t)__popc(ml & window(b));
        }
        if (v < n && !hub) lend[v] = s + nl;
        uint32_t light = s, heavy = s + nl;          // next place of either kind
        for (uint32_t b = 0; b < total; b += 32) {
            const uint32_t j = b + lane;
            const bool valid = j < total;
            const uint32_t own = warp_owner_search(excl, valid ? j : 0);
            const uint32_t at = __shfl_sync(FULL, s - excl, own) + j;
            const uint2 x = valid ? __ldg(&adj[at]) : make_uint2(0, 0);
            const uint32_t ml = __ballot_sync(FULL, valid && x.y < delta);
            const uint32_t w = window(b), lt = lanemask_lt();
            const uint32_t wo = __shfl_sync(FULL, w, own);
            const uint32_t lo = __shfl_sync(FULL, light, own), ho = __shfl_sync(FULL, heavy, own);
            if (valid)
                adj_w[x.y < delta ? lo + __popc(ml & wo & lt) : ho + __popc(~ml & wo & lt)] = x;
            light += (uint32_t)__popc(ml & w);
            heavy += (uint32_t)__popc(~ml & w);
        }
    }
}

constexpr uint32_t PH_THREADS = 512;
constexpr uint32_t PH_PER_THREAD = 8;
__global__ void __launch_bounds__(PH_THREADS) partition_hub_kernel(
    const uint32_t *__restrict__ row_ptr, const uint2 *__restrict__ adj,
    const uint64_t *__restrict__ heavy_chunks, uint32_t n_heavy_chunks, uint32_t delta,
    uint2 *__restrict__ adj_w, uint32_t *__restrict__ lend) {
    constexpr uint32_t TILE = PH_THREADS * PH_PER_THREAD, WARPS = PH_THREADS / 32;
    __shared__ uint32_t wsum[WARPS];
    __shared__ uint32_t hub[32], starts;
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    // 32 chunks at a time; a row is its PART_HUB_DEG / CHUNK-th chunk's
    for (uint32_t i0 = blockIdx.x * 32; i0 < n_heavy_chunks; i0 += gridDim.x * 32) {
        if (w == 0) {
            const uint64_t item = i0 + lane < n_heavy_chunks ? heavy_chunks[i0 + lane] : 0ull;
            hub[lane] = (uint32_t)(item >> 32);
            const uint32_t m = __ballot_sync(FULL, (uint32_t)item == PART_HUB_DEG / CHUNK - 1);
            if (lane == 0) starts = m;
        }
        __syncthreads();
        for (uint32_t m = starts; m; m &= m - 1) {
            const uint32_t v = hub[__ffs(m) - 1], s = row_ptr[v], e = row_ptr[v + 1];
            if (e - s < PART_HUB_DEG) continue;
            uint32_t nl = 0;
#pragma unroll 4
            for (uint64_t j = (uint64_t)s + threadIdx.x; j < e; j += PH_THREADS)
                nl += __ldg(&adj[j].y) < delta;
            nl = __reduce_add_sync(FULL, nl);
            if (lane == 0) wsum[w] = nl;
            __syncthreads();
            nl = 0;
            for (uint32_t k = 0; k < WARPS; ++k) nl += wsum[k];
            __syncthreads();
            if (threadIdx.x == 0) lend[v] = s + nl;
            uint32_t light = s, heavy = s + nl;
            // a thread takes PH_PER_THREAD consecutive arcs of a tile
            for (uint64_t b = s; b < e; b += TILE) {
                const uint64_t j0 = b + threadIdx.x * PH_PER_THREAD;
                uint2 x[PH_PER_THREAD];
                uint32_t mine = 0, have = 0;
#pragma unroll
                for (uint32_t k = 0; k < PH_PER_THREAD; ++k) {
                    x[k] = make_uint2(0, 0);
                    if (j0 + k < e) {
                        x[k] = __ldg(&adj[j0 + k]);
                        mine += x[k].y < delta;
                        ++have;
                    }
                }
                const uint32_t incl = warp_inclusive_scan(mine);
                if (lane == 31) wsum[w] = incl;
                __syncthreads();
                uint32_t before = incl - mine, total = 0;
                for (uint32_t k = 0; k < WARPS; ++k) {
                    if (k < w) before += wsum[k];
                    total += wsum[k];
                }
                __syncthreads();
                uint32_t lo = light + before, ho = heavy + threadIdx.x * PH_PER_THREAD - before;
#pragma unroll
                for (uint32_t k = 0; k < PH_PER_THREAD; ++k)
                    if (k < have) adj_w[x[k].y < delta ? lo++ : ho++] = x[k];
                const uint32_t tile = (uint32_t)min((uint64_t)TILE, e - b);
                light += total;
                heavy += tile - total;
            }
        }
        __syncthreads();
    }
}

cudaError_t launch_partition(const DevGraph &g, uint32_t delta, cudaStream_t s) {
    uint64_t blocks = ((uint64_t)g.n + 255) / 256;
    const uint64_t cap = (uint64_t)current_sm_count() * 32;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    partition_kernel<<<(unsigned)blocks, 256, 0, s>>>(g.row_ptr, g.adj, g.n, delta, g.adj_w, g.lend);
    if (g.n_heavy_chunks) {
        const uint64_t hubs = std::min<uint64_t>(g.n_heavy_chunks, (uint64_t)current_sm_count() * 4);
        partition_hub_kernel<<<(unsigned)hubs, PH_THREADS, 0, s>>>(
            g.row_ptr, g.adj, g.heavy_chunks, g.n_heavy_chunks, delta, g.adj_w, g.lend);
    }
    return cudaGetLastError();
}

cudaError_t ensure_partition_dev(DevGraph &g, uint32_t delta, cudaStream_t s) {
    if (delta > g.max_w || g.m == 0 || g.part_delta == delta) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (!g.adj_w) e = cudaMalloc((void **)&g.adj_w, (size_t)g.m * sizeof(uint2));
    if (e == cudaSuccess && !g.lend) e = cudaMalloc((void **)&g.lend, (size_t)g.n * 4);
    if (e == cudaSuccess) e = launch_partition(g, delta, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        g.part_delta = 0;
        return e;
    }
    g.part_delta = delta;
    return cudaSuccess;
}

cudaError_t launch_validate_graph(const uint32_t *row_ptr, const int32_t *col, const uint32_t *w,
                                  uint32_t n, uint64_t m, uint2 *adj, const uint32_t *new_of,
                                  const uint32_t *new_row_ptr, uint32_t *bad, uint32_t *max_w,
                                  cudaStream_t s) {
    (void)m;
    uint64_t blocks = ((uint64_t)n + 255) / 256;
    const uint64_t cap = (uint64_t)current_sm_count() * 16;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    validate_kernel<<<(unsigned)blocks, 256, 0, s>>>(row_ptr, col, w, n, adj, new_of, new_row_ptr,
                                                      bad, max_w);
    return cudaGetLastError();
}

}  // namespace stn
