// steiner_voronoi_noalloc: Voronoi cells for callers that cannot allocate
// device memory.
//
// Some callers cannot call cudaMalloc at all: code running inside a
// framework that owns every device allocation through its own pool, code
// that must not grow its memory footprint after start-up, or code that has
// to run while the allocator is unavailable.  They already hold the graph
// and the output arrays in device memory of their own.  This entry point
// computes the same per-vertex cell / distance / predecessor as
// steiner_voronoi on such caller-owned arrays, and keeps all of its working
// memory in one fixed file-scope device array (g_scratch below), so it
// allocates nothing: no cudaMalloc, no cudaFree, no allocating library call.
//
// The scratch array exists on every GPU that loads the library, for the
// lifetime of the process, and bounds the graph size (NA_MAX_VERTICES).
// Every call reuses it: a call clears what must start empty and overwrites
// the rest, so calls that overlap on the GPU (other streams, other host
// threads) race with each other and must be serialised by the caller.
//
// One cooperative kernel does the whole call: it clears the state and checks
// the row offsets, seeds the frontier, runs the same packed
// (distance << 32 | seed rank) 64-bit atomicMin fixed point as the library's
// Voronoi path in bands of distance, and derives predecessors and
// writes the outputs, with a grid barrier between the steps.
#include <algorithm>
#include <cstddef>
#include <mutex>
#include <string>

#include "../../include/steiner.h"
#include "common.cuh"

namespace stn {
namespace na {

constexpr uint32_t NA_MAX_VERTICES = STEINER_NOALLOC_MAX_VERTICES;

struct NaControl {
    GridBarrier bar;
    uint32_t err;            // ERR_* bits
    // Rejected input.  The blocks leave together on a word only if nothing
    // writes it after the barrier that they read it behind, so each check has
    // a word of its own: row offsets (written before the first barrier),
    // seeds (between the first and the second), neighbour ids (while the
    // iterations run, read after the last).
    uint32_t bad_rows, bad_seeds, bad_arcs;
    uint32_t count[3];       // frontier: short rows, rotating by iteration
    uint32_t hubs[3];        // frontier: rows of NA_HUB_DEG arcs or more
    uint32_t iterations;
    uint32_t far_min[3];     // smallest distance left beyond the threshold, by phase
    unsigned long long wsum; // sum of the sampled weights
};

// Layout of the scratch array: control block, then per-vertex arrays.
constexpr size_t CTL_BYTES = 256;
constexpr size_t LABEL_OFF = CTL_BYTES;                                   // uint64 [max]
constexpr size_t STAMP_OFF = LABEL_OFF + 8ull * NA_MAX_VERTICES;          // uint32 [max]
constexpr size_t Q0_OFF = STAMP_OFF + 4ull * NA_MAX_VERTICES;             // uint32 [max]
constexpr size_t Q1_OFF = Q0_OFF + 4ull * NA_MAX_VERTICES;                // uint32 [max]
constexpr size_t SCRATCH_BYTES = Q1_OFF + 4ull * NA_MAX_VERTICES;
static_assert(sizeof(NaControl) <= CTL_BYTES, "control block does not fit");

// The only working memory of steiner_voronoi_noalloc (24 MiB + 256 B).
static __device__ __align__(256) unsigned char g_scratch[SCRATCH_BYTES];

struct NaArgs {
    const uint32_t *row_ptr;
    const int32_t *col;
    const uint32_t *w;
    uint32_t n;
    uint64_t n_arcs;
    const int32_t *seeds;
    uint32_t k;
    unsigned char *scratch;     // device address of g_scratch
    uint32_t max_iters;
    uint32_t local_rounds;      // hops a warp follows its own pushes per iteration
    uint32_t sparse;            // few arcs per vertex
    uint32_t banded;            // in bands of distance
    int32_t *cell;
    uint32_t *dist;
    int32_t *pred;
};

__device__ __forceinline__ NaControl *ctl_of(const NaArgs &a) {
    return reinterpret_cast<NaControl *>(a.scratch);
}
__device__ __forceinline__ uint64_t *label_of(const NaArgs &a) {
    return reinterpret_cast<uint64_t *>(a.scratch + LABEL_OFF);
}
__device__ __forceinline__ uint32_t *stamp_of(const NaArgs &a) {
    return reinterpret_cast<uint32_t *>(a.scratch + STAMP_OFF);
}
__device__ __forceinline__ uint32_t *queue_of(const NaArgs &a, uint32_t it) {
    return reinterpret_cast<uint32_t *>(a.scratch + ((it & 1) ? Q1_OFF : Q0_OFF));
}

// Rows of NA_HUB_DEG arcs or more are cut into NA_CHUNK-arc pieces spread
// over the grid's warps; shorter ones are relaxed 32 rows to a warp.
constexpr uint32_t NA_HUB_DEG = 256;
constexpr uint32_t NA_CHUNK = 256;
constexpr int NA_ILP = 4;                  // arcs in flight per lane
constexpr uint32_t NA_WARPS = 8;           // per block
// Band width in mean weights over the mean degree, and what the first band of
// a dense graph is divided by (see the kernel).  Grid 1000 x 1000: 0.90 ms,
// 1.00 at 16, 1.07 at 64, 1.24 without bands; R-MAT of 200,003 vertices: 0.77,
// 0.80 at 16, 0.82 without.
constexpr double NA_BAND = 32;
constexpr uint32_t NA_STEP = 64;
// Dense graphs of fewer arcs run as one band (60,000 vertices, 720,000 arcs:
// 0.26 ms, 0.27 in bands).
constexpr uint64_t NA_BAND_ARCS = 1u << 21;
constexpr uint32_t NA_REGION = 512;        // staged pushes per warp
// Rows of NA_BLOCK_DEG arcs or more take the whole block in the export.
constexpr uint32_t NA_BLOCK_DEG = 1024;

// A frontier: short rows from the bottom of its queue, hubs from the top
// (a vertex is queued once, so the two never meet).
struct NaFront {
    uint32_t *q;
    uint32_t *count, *hubs;
    uint32_t tag;
};

__device__ __forceinline__ void na_queue(const NaArgs &a, const NaFront &f, bool want, uint32_t v,
                                         uint32_t *err) {
    bool hub = false;
    if (want) {
        want = atomicExch(&stamp_of(a)[v], f.tag) != f.tag;
        hub = a.row_ptr[v + 1] - a.row_ptr[v] >= NA_HUB_DEG;
    }
    uint32_t g = warp_append(want && !hub, f.count, a.n, err);
    if (g != INF32) f.q[g] = v;
    g = warp_append(want && hub, f.hubs, a.n, err);
    if (g != INF32) f.q[a.n - 1 - g] = v;
}

// Stages v in the warp's region, or queues it when that is full.
__device__ __forceinline__ void na_stage(const NaArgs &a, const NaFront &f, uint32_t *region,
                                         uint32_t *region_n, bool want, uint32_t v, uint32_t *err) {
    const uint32_t mask = __ballot_sync(FULL, want);
    if (mask == 0) return;
    const uint32_t n = *(volatile uint32_t *)region_n;
    const uint32_t slot = n + (uint32_t)__popc(mask & lanemask_lt());
    if (want && slot < NA_REGION) region[slot] = v;
    __syncwarp();
    if (lane_id() == 0) *(volatile uint32_t *)region_n = min(n + (uint32_t)__popc(mask), NA_REGION);
    __syncwarp();
    if (n + (uint32_t)__popc(mask) > NA_REGION) na_queue(a, f, want && slot >= NA_REGION, v, err);
}

// Relaxes up to NA_ILP arcs per lane (arc index and tail label each), the
// loads and atomics of all of them issued back to back; vertices that
// improve are staged in the warp's region (a vertex may be staged twice),
// or queued when it is full.
__device__ __forceinline__ void na_relax(const NaArgs &a, NaControl *c, const NaFront &f,
                                         uint32_t *region, uint32_t *region_n,
                                         const bool (&valid)[NA_ILP],
                                         const uint32_t (&arc)[NA_ILP],
                                         const uint64_t (&lab)[NA_ILP], uint32_t T,
                                         uint32_t &fmin) {
    uint64_t *label = label_of(a);
    int32_t cv[NA_ILP];
    uint32_t wt[NA_ILP];
#pragma unroll
    for (int i = 0; i < NA_ILP; ++i) {
        cv[i] = -1;
        wt[i] = 0;
        if (valid[i]) {
            cv[i] = a.col[arc[i]];
            wt[i] = a.w[arc[i]];
        }
    }
    uint64_t nl[NA_ILP], cur[NA_ILP];
    bool imp[NA_ILP];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < NA_ILP; ++i) {
        nl[i] = INF64;
        cur[i] = 0;
        if (!valid[i]) continue;
        if (cv[i] < 0 || (uint32_t)cv[i] >= a.n) {
            bad = true;
            continue;
        }
        const uint64_t nd = (lab[i] >> 32) + (uint64_t)wt[i];
        if (nd < INF32) {          // the export reports a distance beyond
            nl[i] = (nd << 32) | (lab[i] & 0xFFFFFFFFull);
            cur[i] = ldcg_u64(&label[cv[i]]);
        }
    }
    if (bad) atomicOr(&c->bad_arcs, 1u);
#pragma unroll
    for (int i = 0; i < NA_ILP; ++i) {
        imp[i] = false;
        if (nl[i] < cur[i])
            imp[i] = nl[i] < atomicMin(reinterpret_cast<unsigned long long *>(&label[cv[i]]),
                                       (unsigned long long)nl[i]);
        if (imp[i] && (uint32_t)(nl[i] >> 32) >= T) {    // waits for its band
            fmin = min(fmin, (uint32_t)(nl[i] >> 32));
            imp[i] = false;
        }
    }
    if (!__any_sync(FULL, imp[0] | imp[1] | imp[2] | imp[3])) return;
#pragma unroll
    for (int i = 0; i < NA_ILP; ++i) na_stage(a, f, region, region_n, imp[i], (uint32_t)cv[i], &c->err);
}

// Relaxes the rows of up to 32 vertices (has, u: one per lane), their arcs
// flattened over the lanes.  Hubs are left to the hub pass of the next
// iteration (`requeue`) or were queued as such.
__device__ __forceinline__ void na_relax_rows(const NaArgs &a, NaControl *c, const NaFront &f,
                                              uint32_t *region, uint32_t *region_n, bool has,
                                              uint32_t u, bool requeue, uint32_t T,
                                              uint32_t &fmin) {
    const uint32_t lane = lane_id();
    uint32_t s = 0, deg = 0;
    uint64_t lab = INF64;
    if (has) {
        s = a.row_ptr[u];
        deg = a.row_ptr[u + 1] - s;
        lab = ldcg_u64(&label_of(a)[u]);
    }
    if (requeue) {
        const bool hub = deg >= NA_HUB_DEG;
        if (__any_sync(FULL, hub)) na_queue(a, f, hub, u, &c->err);
        if (hub) deg = 0;
    }
    const uint32_t incl = warp_inclusive_scan(deg);
    const uint32_t excl = incl - deg;
    const uint32_t total = __shfl_sync(FULL, incl, 31);
    for (uint32_t b = 0; b < total; b += 32 * NA_ILP) {
        bool valid[NA_ILP];
        uint32_t arc[NA_ILP];
        uint64_t labs[NA_ILP];
#pragma unroll
        for (int i = 0; i < NA_ILP; ++i) {
            const uint32_t j = b + lane + 32 * i;
            valid[i] = j < total;
            const uint32_t owner = warp_owner_search(excl, valid[i] ? j : 0);
            const uint32_t so = __shfl_sync(FULL, s, owner);
            const uint32_t eo = __shfl_sync(FULL, excl, owner);
            labs[i] = __shfl_sync(FULL, lab, owner);
            arc[i] = so + (j - eo);
        }
        na_relax(a, c, f, region, region_n, valid, arc, labs, T, fmin);
    }
}

// pred(v) = smallest-id tight neighbour in v's cell: the first tight arc of
// the row.  Arc `e` of reached vertex v: its index if tight, else INF32; a
// reached vertex next to an unreached one means a distance did not fit below
// 2^32 - 1.
__device__ __forceinline__ uint32_t na_tight(const NaArgs &a, uint64_t lv, uint32_t e,
                                             bool &overflow) {
    const int32_t cu = a.col[e];
    const uint32_t wt = a.w[e];
    if (cu < 0 || (uint32_t)cu >= a.n) return INF32;
    const uint64_t lu = ldcg_u64(&label_of(a)[cu]);
    if (lu == INF64) {
        overflow = true;
        return INF32;
    }
    return (uint32_t)lu == (uint32_t)lv && (lu >> 32) + wt == lv >> 32 ? e : INF32;
}

__device__ __forceinline__ void na_write(const NaArgs &a, uint32_t v, uint64_t lv, uint32_t arc) {
    const bool reached = lv != INF64;
    if (a.cell) a.cell[v] = reached ? a.seeds[(uint32_t)lv] : -1;
    if (a.dist) a.dist[v] = reached ? (uint32_t)(lv >> 32) : INF32;
    if (a.pred) a.pred[v] = !reached ? -1 : (lv >> 32) == 0 ? (int32_t)v
                                          : arc != INF32 ? a.col[arc] : -1;
}

// The whole call.  What bounds it: on small-world graphs the relaxations of
// a few thick iterations (23 G arcs per second; hub rows are cut over the
// grid), on
// high-diameter ones the chain of hops, a barrier each; local_rounds lets a
// warp follow its own pushes several hops between barriers.
// R-MAT of 200,003 vertices, k = 300: 0.77 ms (12.7 with a hub's row walked
// by one warp, and by one thread for its predecessor); grid 499 x 401,
// k = 25: 0.62-0.97 ms (3.5 with a barrier per hop of 1216 blocks).
__global__ void __launch_bounds__(256, 4) na_kernel(NaArgs a) {
    __shared__ uint32_t region_s[NA_WARPS][NA_REGION];
    __shared__ uint32_t region_n_s[NA_WARPS];
    __shared__ uint32_t first_s[NA_WARPS][32];      // export: first tight arc per row
    __shared__ uint32_t big_s[256], big_n, big_arc;
    __shared__ uint32_t hub_s[256], hub_deg_s[256];
    __shared__ uint64_t hub_lab_s[256];
    NaControl *c = ctl_of(a);
    uint64_t *label = label_of(a);
    const uint32_t lane = lane_id(), wib = threadIdx.x >> 5;
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
    const uint32_t warp = gtid >> 5, nwarps = nth >> 5;
    const bool first = gtid == 0;
    uint32_t *region = region_s[wib], *region_n = &region_n_s[wib];
    uint32_t bar_target = 0;

    // Clear the previous call's state; check the row offsets (row_ptr[0] =
    // 0, non-decreasing, row_ptr[n] = n_arcs), so that no arc outside
    // [0, n_arcs) is read later.
    {
        bool bad = first && (a.row_ptr[0] != 0 || (uint64_t)a.row_ptr[a.n] != a.n_arcs);
        uint32_t *stamp = stamp_of(a);
        for (uint32_t v = gtid; v < a.n; v += nth) {
            label[v] = INF64;
            stamp[v] = 0;
            bad |= a.row_ptr[v] > a.row_ptr[v + 1];
        }
        if (bad) atomicOr(&c->bad_rows, 1u);
        if (first) c->far_min[0] = c->far_min[1] = c->far_min[2] = INF32;
    }
    if (!grid_sync(&c->bar, &c->err, bar_target)) return;
    if (ldcg_u32(&c->bad_rows)) return;
    // One weight per thread, spread evenly over the arcs (only now: the arc
    // count is known to be the row offsets').
    {
        unsigned long long wt = a.n_arcs ? a.w[a.n_arcs * gtid / nth] : 0u;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) wt += __shfl_xor_sync(FULL, wt, o);
        if (lane == 0) atomicAdd(&c->wsum, wt);
    }
    // Seeds (ascending, distinct, in range) at distance 0 on the first
    // frontier (iteration 0, tag 1).
    for (uint32_t r0 = warp * 32; r0 < a.k; r0 += nwarps * 32) {
        const uint32_t r = r0 + lane;
        int32_t s = 0;
        bool ok = r < a.k;
        if (ok) {
            s = a.seeds[r];
            if (s < 0 || (uint32_t)s >= a.n || (r && a.seeds[r - 1] >= s)) {
                atomicOr(&c->bad_seeds, 1u);
                ok = false;
            } else {
                label[s] = (uint64_t)r;
            }
        }
        na_queue(a, NaFront{queue_of(a, 0), &c->count[0], &c->hubs[0], 1u}, ok, (uint32_t)s, &c->err);
    }
    if (!grid_sync(&c->bar, &c->err, bar_target)) return;
    if (ldcg_u32(&c->bad_seeds)) return;

    // Iteration `it` relaxes the arcs of its frontier, queueing every vertex
    // whose label drops below the threshold T (once per iteration, by stamp).
    // When the frontier is thin the threshold goes up by a band, and the next
    // iteration first reads all labels for the vertices between the two (no
    // pile is kept: reading 8 n bytes costs less than a barrier).
    // Every block decides on counts that no iteration writes before all have
    // read them, and a thin frontier always ends the phase, so that the
    // minimum left beyond T is complete too.
    uint32_t nf = min(ldcg_u32(&c->count[0]), a.n), nh = min(ldcg_u32(&c->hubs[0]), a.n);
    const double mean = (double)ldcg_u64(reinterpret_cast<const uint64_t *>(&c->wsum)) / nth;
    const double width = NA_BAND * mean * a.n / (double)max((unsigned long long)a.n_arcs, 1ull);
    const uint32_t delta = width >= 4e9 ? 4000000000u : width < 1 ? 1u : (uint32_t)width;
    uint32_t T = a.sparse ? delta : a.banded ? max(1u, delta / NA_STEP) : INF32, T_old = T;
    uint32_t band = delta;
    const uint32_t thin = a.sparse ? 8 * nwarps : nwarps;
    uint32_t phase = 0;
    bool split = false;
    for (uint32_t it = 0;; ++it) {
        if (first) c->count[(it + 2) % 3] = c->hubs[(it + 2) % 3] = 0;
        const uint32_t *qc = queue_of(a, it);
        const NaFront f{queue_of(a, it + 1), &c->count[(it + 1) % 3], &c->hubs[(it + 1) % 3], it + 2};
        if (lane == 0) *region_n = 0;
        __syncwarp();
        uint32_t fmin = INF32;
        if (split) {
            for (uint32_t b = warp * 32; b < a.n; b += nwarps * 32) {
                const uint32_t v = b + lane;
                const uint32_t d = v < a.n ? (uint32_t)(ldcg_u64(&label[v]) >> 32) : INF32;
                if (d >= T) fmin = min(fmin, d);
                na_stage(a, f, region, region_n, d >= T_old && d < T, v, &c->err);
            }
        }
        // hubs: 256 at a time, loaded one per thread of the block, then seen
        // by each of its warps; piece p of hub h goes to warp (p + 97 h) mod
        // nwarps (loaded 32 at a time by every warp, the chain of loads over
        // a few thousand hubs was most of a thick iteration: R-MAT of 2^20
        // vertices 3.8 -> 3.3 ms)
        for (uint32_t h0 = 0; h0 < nh; h0 += 256) {
            if (h0) __syncthreads();
            hub_deg_s[threadIdx.x] = 0;
            if (h0 + threadIdx.x < nh) {
                const uint32_t u = ldcg_u32(&qc[a.n - 1 - (h0 + threadIdx.x)]);
                const uint32_t r0 = a.row_ptr[u];
                hub_s[threadIdx.x] = r0;
                hub_deg_s[threadIdx.x] = a.row_ptr[u + 1] - r0;
                hub_lab_s[threadIdx.x] = ldcg_u64(&label[u]);
            }
            __syncthreads();
            for (uint32_t g = 0; g < 256 && h0 + g < nh; g += 32) {
                const uint32_t s = hub_s[g + lane], deg = hub_deg_s[g + lane];
                const uint64_t lab = hub_lab_s[g + lane];
                const uint32_t pieces = deg / NA_CHUNK + (deg % NA_CHUNK != 0);
                const uint32_t p0 = (warp + nwarps - (h0 + g + lane) * 97u % nwarps) % nwarps;
                for (uint32_t m = __ballot_sync(FULL, p0 < pieces); m; m &= m - 1) {
                    const uint32_t l = __ffs(m) - 1;
                    const uint32_t sl = __shfl_sync(FULL, s, l), dl = __shfl_sync(FULL, deg, l);
                    const uint64_t ll = __shfl_sync(FULL, lab, l);
                    for (uint64_t p = __shfl_sync(FULL, p0, l); p * NA_CHUNK < dl; p += nwarps) {
                        const uint32_t lo = (uint32_t)p * NA_CHUNK, hi = lo + min(dl - lo, NA_CHUNK);
                        // (steps counted from the piece's start: in a row of almost
                        // 2^32 arcs b and j may wrap, to arcs of the same row)
                        for (uint32_t h = 0; h < NA_CHUNK; h += 32 * NA_ILP) {
                            const uint32_t b = lo + h;
                            if (b >= hi) break;
                            bool valid[NA_ILP];
                            uint32_t arc[NA_ILP];
                            uint64_t labs[NA_ILP];
#pragma unroll
                            for (int i = 0; i < NA_ILP; ++i) {
                                const uint32_t j = b + lane + 32 * i;
                                valid[i] = j < hi;
                                arc[i] = sl + j;
                                labs[i] = ll;
                            }
                            na_relax(a, c, f, region, region_n, valid, arc, labs, T, fmin);
                        }
                    }
                }
            }
        }
        // short rows: a thin frontier is spread over all warps
        const uint32_t per = (nf + nwarps - 1) / nwarps;
        const uint32_t bsz = per <= 1 ? 1 : per <= 2 ? 2 : per <= 4 ? 4 : per <= 8 ? 8 : per <= 16 ? 16 : 32;
        for (uint32_t b0 = warp * bsz; b0 < nf; b0 += nwarps * bsz) {
            const bool has = lane < bsz && b0 + lane < nf;
            const uint32_t u = has ? ldcg_u32(&qc[b0 + lane]) : 0;
            na_relax_rows(a, c, f, region, region_n, has, u, false, T, fmin);
        }
        // the warp follows its own pushes, a hop per round
        uint32_t lo = 0;
        const uint32_t rounds = nf + nh < thin ? a.local_rounds : 0u;
        for (uint32_t r = 0; r < rounds; ++r) {
            __syncwarp();
            const uint32_t hi = *(volatile uint32_t *)region_n;
            if (lo >= hi || hi - lo > 32) break;
            for (uint32_t b0 = lo; b0 < hi; b0 += 32) {
                const bool has = b0 + lane < hi;
                na_relax_rows(a, c, f, region, region_n, has, has ? region[b0 + lane] : 0, true, T, fmin);
            }
            lo = hi;
        }
        __syncwarp();
        const uint32_t staged = *(volatile uint32_t *)region_n;
        for (uint32_t b0 = lo; b0 < staged; b0 += 32) {
            const bool has = b0 + lane < staged;
            na_queue(a, f, has, has ? region[b0 + lane] : 0, &c->err);
        }
        fmin = __reduce_min_sync(FULL, fmin);
        if (lane == 0 && fmin != INF32) atomicMin(&c->far_min[phase % 3], fmin);
        if (!grid_sync(&c->bar, &c->err, bar_target)) return;
        if (it + 1 >= a.max_iters) {
            if (first) atomicOr(&c->err, ERR_TIMEOUT);
            return;
        }
        nf = min(ldcg_u32(&c->count[(it + 1) % 3]), a.n);
        nh = min(ldcg_u32(&c->hubs[(it + 1) % 3]), a.n);
        split = false;
        if (nf + nh >= thin) continue;
        const uint32_t next = ldcg_u32(&c->far_min[phase % 3]);
        if ((nf | nh) == 0 && next == INF32) {
            if (first) c->iterations = it + 1;
            break;
        }
        ++phase;
        if (first) c->far_min[(phase + 1) % 3] = INF32;    // last read a phase ago, next used a phase from now
        if (next != INF32) {
            T_old = T;
            // (bands that hold next to nothing widen: on a path each would end
            // an iteration early; 537 ms for 10^6 vertices against 613)
            band = a.sparse && nf + nh < nwarps / 8 ? min(2 * (uint64_t)band, (uint64_t)0x80000000u) : delta;
            T = (uint32_t)min((uint64_t)INF32, (uint64_t)max(T, next) + band);
            split = true;
        }
    }

    // Predecessors and outputs in the steiner_voronoi format.  A rejected
    // input leaves the caller's outputs untouched.  A block takes 256 rows,
    // a warp 32 of them with their arcs flattened over its lanes; rows of
    // NA_BLOCK_DEG arcs or more are then scanned by the whole block.
    if (ldcg_u32(&c->bad_arcs)) return;
    bool overflow = false;
    for (uint32_t v0 = blockIdx.x * 256; v0 < a.n; v0 += gridDim.x * 256) {
        if (threadIdx.x == 0) big_n = 0;
        first_s[wib][lane] = INF32;
        __syncthreads();
        const uint32_t v = v0 + threadIdx.x;
        uint32_t s = 0, deg = 0;
        uint64_t lv = INF64;
        bool big = false;
        if (v < a.n) {
            lv = ldcg_u64(&label[v]);
            if (lv != INF64) {
                s = a.row_ptr[v];
                deg = a.row_ptr[v + 1] - s;
                big = deg >= NA_BLOCK_DEG;
            }
        }
        if (big) {
            big_s[atomicAdd(&big_n, 1u)] = v;
            deg = 0;
        }
        const uint32_t incl = warp_inclusive_scan(deg);
        const uint32_t excl = incl - deg;
        const uint32_t total = __shfl_sync(FULL, incl, 31);
        for (uint32_t b = 0; b < total; b += 32 * NA_ILP) {
#pragma unroll
            for (int i = 0; i < NA_ILP; ++i) {
                const uint32_t j = b + lane + 32 * i;
                const uint32_t owner = warp_owner_search(excl, j < total ? j : 0);
                const uint32_t so = __shfl_sync(FULL, s, owner), eo = __shfl_sync(FULL, excl, owner);
                const uint64_t lo = __shfl_sync(FULL, lv, owner);
                if (j >= total) continue;
                const uint32_t t = na_tight(a, lo, so + (j - eo), overflow);
                if (t != INF32) atomicMin(&first_s[wib][owner], t);
            }
        }
        __syncwarp();
        if (v < a.n && !big) na_write(a, v, lv, first_s[wib][lane]);
        __syncthreads();
        for (uint32_t i = 0; i < big_n; ++i) {
            const uint32_t u = big_s[i];
            if (threadIdx.x == 0) big_arc = INF32;
            __syncthreads();
            const uint64_t lu = ldcg_u64(&label[u]);
            const uint32_t r1 = a.row_ptr[u + 1];
            uint32_t best = INF32;
            // (64-bit: a row may end next to 2^32)
            for (uint64_t e0 = (uint64_t)a.row_ptr[u] + threadIdx.x; e0 < r1; e0 += 256 * NA_ILP) {
#pragma unroll
                for (int q = 0; q < NA_ILP; ++q) {
                    const uint64_t e = e0 + 256u * q;
                    if (e < r1) best = min(best, na_tight(a, lu, (uint32_t)e, overflow));
                }
            }
            best = __reduce_min_sync(FULL, best);
            if (lane == 0 && best != INF32) atomicMin(&big_arc, best);
            __syncthreads();
            if (threadIdx.x == 0) na_write(a, u, lu, big_arc);
        }
        __syncthreads();
    }
    if (__any_sync(FULL, overflow) && lane == 0) atomicOr(&c->err, ERR_OVERFLOW);
}

// Per-device set-up: the device address of g_scratch (host code cannot use
// the symbol itself) and the cooperative grid size.
struct DeviceSetup {
    bool ready = false;
    unsigned char *scratch = nullptr;
    int blocks = 0;
    int sms = 0;
};
constexpr int NA_MAX_DEVICES = 64;
static DeviceSetup g_setup[NA_MAX_DEVICES];
static std::mutex g_setup_mu;

static int setup_device(int dev, DeviceSetup &out, const char **why) {
    std::lock_guard<std::mutex> lk(g_setup_mu);
    DeviceSetup &s = g_setup[dev];
    if (!s.ready) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_scratch);
        if (e != cudaSuccess) {
            *why = cudaGetErrorString(e);
            return STEINER_ECUDA;
        }
        int per_sm = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, na_kernel, 256, 0);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess || per_sm < 1) {
            *why = e != cudaSuccess ? cudaGetErrorString(e) : "kernel does not fit on an SM";
            return STEINER_ECUDA;
        }
        s.scratch = static_cast<unsigned char *>(ptr);
        s.blocks = per_sm * sms;
        s.sms = sms;
        s.ready = true;
    }
    out = s;
    return STEINER_OK;
}

}  // namespace na

void api_set_error(const std::string &msg);

}  // namespace stn

using namespace stn;
using namespace stn::na;

extern "C" int steiner_voronoi_noalloc(const uint32_t *row_ptr, const int32_t *col,
                                       const uint32_t *w, uint32_t n, uint64_t n_arcs,
                                       const int32_t *seeds, uint32_t k, int32_t *cell,
                                       uint32_t *dist, int32_t *pred, void *stream) {
    if (n > NA_MAX_VERTICES) {
        api_set_error("steiner_voronoi_noalloc: n exceeds its fixed scratch limit of "
                      "STEINER_NOALLOC_MAX_VERTICES (1048576) vertices");
        return STEINER_ENOMEM;
    }
    if (n == 0 || k == 0 || k > n || !row_ptr || !seeds || (n_arcs && (!col || !w)) ||
        n_arcs >= 0xFFFFFFFFull) {
        api_set_error("steiner_voronoi_noalloc: invalid arguments");
        return STEINER_EINVAL;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
        api_set_error("steiner_voronoi_noalloc: no usable current device");
        return STEINER_ECUDA;
    }
    DeviceSetup su;
    const char *why = "";
    int rc = setup_device(dev, su, &why);
    if (rc) {
        api_set_error(std::string("steiner_voronoi_noalloc set-up: ") + why);
        return rc;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // A warp per 256 arcs or 32 vertices and at least one block: a small
    // graph's iterations end at a barrier of fewer blocks.  Graphs of few
    // arcs per vertex have a high diameter (grids, paths, trees): there a
    // warp follows its own pushes up to 16 hops between barriers.
    const uint64_t warps = std::max<uint64_t>(n_arcs / 256, (n + 31) / 32);
    const unsigned blocks = (unsigned)std::min<uint64_t>((warps + 7) / 8, (uint64_t)su.blocks);
    const uint32_t sparse = n_arcs <= 8ull * n ? 1u : 0u;
    NaArgs a{row_ptr, col, w, n, n_arcs, seeds, k, su.scratch, 1u << 22,
             sparse ? 16u : 0u, sparse, sparse || n_arcs >= NA_BAND_ARCS ? 1u : 0u, cell, dist, pred};
    e = cudaMemsetAsync(su.scratch, 0, sizeof(NaControl), s);
    if (e == cudaSuccess) {
        void *args[] = {&a};
        e = cudaLaunchCooperativeKernel((const void *)na_kernel, dim3(blocks), dim3(256), args, 0, s);
    }
    struct {
        uint32_t err, bad_rows, bad_seeds, bad_arcs;
    } r = {};
    static_assert(offsetof(NaControl, bad_arcs) == offsetof(NaControl, err) + 12, "read back as one");
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&r, su.scratch + offsetof(NaControl, err), sizeof(r),
                            cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        api_set_error(std::string("steiner_voronoi_noalloc: ") + cudaGetErrorString(e));
        return STEINER_ECUDA;
    }
    if (r.bad_rows | r.bad_seeds | r.bad_arcs) {
        api_set_error("steiner_voronoi_noalloc: seeds must be distinct, ascending and below n, "
                      "row_ptr must run from 0 to n_arcs without decreasing, and every "
                      "neighbour id must be below n");
        return STEINER_EINVAL;
    }
    if (r.err & (ERR_BARRIER | ERR_TIMEOUT)) {
        api_set_error("steiner_voronoi_noalloc: device loop or barrier hit its cap");
        return STEINER_ETIMEOUT;
    }
    if (r.err & ERR_OVERFLOW) {
        api_set_error("steiner_voronoi_noalloc: a distance reached 2^32 - 1");
        return STEINER_EOVERFLOW;
    }
    if (r.err & ERR_CAPACITY) {
        api_set_error("steiner_voronoi_noalloc: frontier capacity exceeded");
        return STEINER_ENOMEM;
    }
    return STEINER_OK;
}
