// One pass over every arc after the Voronoi fixed point, fusing two steps:
//
//  * pred (Algorithm 2 Step 1's predecessor state; Algorithm 4 line 8):
//    pred(v) = the smallest-id neighbour u with cell(u) = cell(v) and
//    d1(u) + d(u,v) = d1(v).  Rows are sorted by neighbour id, so the
//    smallest arc index in v's row is the smallest id: atomicMin on the
//    arc index.
//  * bridges (Algorithm 2 Step 2; Algorithm 5): for an arc u -> v with
//    rank(cell u) < rank(cell v), b = d1(u) + d(u,v) + d1(v); the pair's
//    table slot keeps min((b << 32) | arc) by 64-bit atomicMin, which is
//    the minimum bridge with the smallest arc id among ties.  This single
//    table stands in for the paper's per-partition maps plus its
//    MPI_Allreduce(MIN) (GLOBAL_MIN_DIST_EDGE_COLL).
//
// The pair table is a direct-address table over the k(k-1)/2 seed pairs
// (an upper-triangle index, i.e. a collision-free hash of the pair).
//
// Load balance: vertices with degree < HEAVY_DEG are processed 32 per warp
// with their arcs flattened over the lanes (labels of 32 consecutive
// vertices are one coalesced load), in the vertex ranges of about equal
// arcs that the dense frontiers use; higher-degree rows are split into
// CHUNK-arc pieces listed once at graph load (smaller ones while they are
// too few for the grid).  With 32 consecutive rows to a warp the first
// batches after the hubs held up to 32 x 255 arcs, read 32 at a time: pairs
// and predecessors of R-MAT 16 took 0.19 ms, 0.034 in ranges; R-MAT of 10^6
// vertices 0.26 against 0.14; R-MAT 26 (degree 8) 5.9 against 5.6.
#include <algorithm>

#include "internal.h"

namespace stn {

// Pieces of a hub chunk while chunks are few: 128 arcs, four steps.
constexpr uint32_t SCAN_SUBS = 4;

struct ScanArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;
    const uint64_t *__restrict__ heavy_chunks;
    uint32_t n_heavy_chunks;
    uint32_t subs;                   // pieces a chunk is cut into (1 or SCAN_SUBS)
    const uint32_t *__restrict__ items;   // vertex ranges [items[i], items[i + 1])
    uint32_t n_items;
    uint32_t n;
    const uint64_t *label;
    const uint32_t *label32;         // narrow labels (the narrow kernel)
    uint32_t lshift;
    uint32_t *pred_arc;
    uint64_t *pairtab;
    uint32_t k;
    bool pairs;
    uint32_t *err;
    const uint32_t *orig_of;         // internal -> caller ids (null: identity)
    const uint32_t *orig_row_ptr;
};

// Label of v in the 64-bit form.
template <bool NARROW>
__device__ __forceinline__ uint64_t scan_label(const ScanArgs &a, uint32_t v) {
    if (NARROW) return widen_label(__ldg(&a.label32[v]), a.lshift);
    return __ldg(reinterpret_cast<const unsigned long long *>(&a.label[v]));
}

// Arc `arc` of row v.  The bridge key carries the caller's arc index,
// cbase + arc (cbase: the caller's row start of v minus v's internal row
// start, taken once per row), so ties between equal bridges break on the
// caller's CSR order whatever the internal vertex order.
template <bool NARROW>
__device__ __forceinline__ void scan_arc(const ScanArgs &a, bool valid, uint32_t v, uint64_t lv,
                                         uint32_t cbase, uint32_t arc, uint2 e, bool &overflow) {
    if (!valid) return;
    uint64_t lu = scan_label<NARROW>(a, e.x);
    if (lv == INF64 || lu == INF64) {
        // a reached vertex next to an unreached one: its true distance is
        // finite but did not fit below 2^32 - 1
        if (lv != lu) overflow = true;
        return;
    }
    uint32_t cv = (uint32_t)lv, cu = (uint32_t)lu;
    uint64_t dv = lv >> 32, du = lu >> 32;
    if (cu == cv) {
        if (du + e.y == dv) atomicMin(&a.pred_arc[v], arc);
    } else if (a.pairs && cv < cu) {
        uint64_t b = dv + e.y + du;
        if (b >= INF32) {
            overflow = true;
            return;
        }
        uint64_t key = (b << 32) | (uint32_t)(cbase + arc);
        uint64_t *slot = &a.pairtab[pair_slot(cv, cu, a.k)];
        // a cached read may be stale, i.e. larger: at worst one atomic more
        if (key < __ldg(reinterpret_cast<const unsigned long long *>(slot)))
            atomicMin(reinterpret_cast<unsigned long long *>(slot), (unsigned long long)key);
    }
}

template <bool NARROW>
__global__ void __launch_bounds__(256) scan_kernel(ScanArgs a) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_hub = a.n_heavy_chunks * a.subs;
    const uint32_t n_work = n_hub + a.n_items;
    bool overflow = false;
    for (uint32_t wi = warp; wi < n_work; wi += nwarps) {
        if (wi < n_hub) {
            uint64_t item = a.heavy_chunks[wi / a.subs];
            uint32_t v = (uint32_t)(item >> 32), c = (uint32_t)item;
            uint32_t rs = a.row_ptr[v];
            const RowPiece p = row_piece(rs, a.row_ptr[v + 1], c * CHUNK + wi % a.subs * (CHUNK / SCAN_SUBS),
                                         CHUNK / a.subs);
            if (p.count == 0) continue;
            uint64_t lv = scan_label<NARROW>(a, v);
            uint32_t cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, v, rs);
            // the next 32 arcs' records are loaded while these are scanned
            uint2 en = make_uint2(0, 0);
            if (lane < p.count) en = __ldcs(&a.adj[p.first + lane]);    // streamed once: evict first
            for (uint32_t j = lane; j < p.count + lane; j += 32) {
                const uint2 ec = en;
                if (j + 32 < p.count) en = __ldcs(&a.adj[p.first + j + 32]);
                scan_arc<NARROW>(a, j < p.count, v, lv, cbase, p.first + j, ec, overflow);
            }
            continue;
        }
        const uint32_t v1 = __ldg(&a.items[wi - n_hub + 1]);
        for (uint32_t vb = __ldg(&a.items[wi - n_hub]); vb < v1; vb += 32) {
            uint32_t v = vb + lane;
            uint32_t s = 0, deg = 0, cbase = 0;
            uint64_t lv = INF64;
            if (v < v1) {
                s = a.row_ptr[v];
                deg = a.row_ptr[v + 1] - s;
                if (deg >= HEAVY_DEG) deg = 0;          // covered by the chunk list
                lv = scan_label<NARROW>(a, v);
                if (deg) cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, v, s);
            }
            uint32_t incl = warp_inclusive_scan(deg);
            uint32_t excl = incl - deg;
            uint32_t total = __shfl_sync(FULL, incl, 31);
            // arc j of the batch belongs to the lane whose prefix covers it;
            // the next 32 arcs' records are loaded while these are scanned
            uint32_t own = warp_owner_search(excl, lane < total ? lane : 0);
            const uint32_t s0 = __shfl_sync(FULL, s, own), x0 = __shfl_sync(FULL, excl, own);
            uint2 en = make_uint2(0, 0);
            if (lane < total) en = __ldcs(&a.adj[s0 + (lane - x0)]);
            for (uint32_t b = 0; b < total; b += 32) {
                const uint32_t j = b + lane;
                const bool valid = j < total;
                const uint32_t owner = own;
                const uint32_t arc = __shfl_sync(FULL, s, owner) + (j - __shfl_sync(FULL, excl, owner));
                const uint2 ec = en;
                const uint32_t jn = j + 32;
                own = warp_owner_search(excl, jn < total ? jn : 0);
                const uint32_t sn = __shfl_sync(FULL, s, own), xn = __shfl_sync(FULL, excl, own);
                if (jn < total) en = __ldcs(&a.adj[sn + (jn - xn)]);
                const uint64_t lo = __shfl_sync(FULL, lv, owner);
                const uint32_t co = __shfl_sync(FULL, cbase, owner);
                const uint32_t vo = vb + owner;
                scan_arc<NARROW>(a, valid, vo, lo, co, arc, ec, overflow);
            }
        }
    }
    if (__any_sync(FULL, overflow) && lane == 0) atomicOr(a.err, ERR_OVERFLOW);
}

// ---------------------------------------------------------------------------
// the scan of a query that returns the tree alone
// ---------------------------------------------------------------------------
//
// A tree needs the MST of G'_1, not all of G'_1, and the predecessors of its
// own vertices.  With rows split at band width delta, most arcs of a large
// graph join cells that bridges lighter than delta have joined already:
//
//  1. tree_scan_kernel reads the light part of the rows of the vertices nearer
//     than delta: every pair of cells with a bridge below delta gets its
//     minimum (such a bridge's arc is lighter than delta, its ends nearer),
//     and these vertices their predecessors (a tight arc is no heavier than
//     its head's distance).  Hub rows farther out are read for the
//     predecessor alone; the predecessors of the other vertices beyond delta
//     are found by the expansion, for those on the tree.
//  2. The MST of those pairs is the part of Kruskal's tree below delta.  Of
//     its components the one whose cells hold the most arcs (sampled) is the
//     hub component.
//  3. rest_scan_kernel reads the rows of the vertices outside the hub
//     component's cells.  Every arc between two components has such an end,
//     so the minimum bridge of every pair of cells in different components is
//     now in the table; pairs inside a component are joined by the
//     component's own tree, by bridges below delta, and cannot add to it.
//  4. The MST of all pairs in the table is then the MST of G'_1.
//
// A bridge key carries the caller's index of its arc, which a row split by
// weight does not give: it is searched in the id-ordered row, for proposals
// that lower the table (first with an index above all, so that few others
// search).  Narrow labels only: their distances rule out an overflow.
// Bound by the label gathers and, at k = 10,000, by probes of a 400 MB table:
// looking at every bridge in step 1, and at every arc of the vertices beyond
// delta, took it 1.91 ms on R-MAT 26 (degree 8) against 1.08.
// Where few bridges are lighter than delta the rest scan reads most rows:
// proposing an arc between two cells from the cell of larger rank only where
// the other's row is not read, and turning ties away before the search, took
// a query of R-MAT 24 (weights to 20, delta 2, k = 10,000) from 11.4 to 8.3 ms.

struct TreeScanArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;       // rows in the caller's order
    const uint2 *__restrict__ adj_w;     // rows with the light arcs first
    const uint32_t *__restrict__ lend;   // end of the light part
    const uint64_t *__restrict__ heavy_chunks;
    uint32_t n_heavy_chunks;
    const uint32_t *__restrict__ items;
    uint32_t n_items;
    uint32_t delta;
    uint32_t near;                       // smallest label of a distance delta
    const uint32_t *label32;
    uint32_t lshift;
    uint32_t *pred_arc;                  // index in adj_w (vertex nearer than delta) or adj
    uint64_t *pairtab;
    uint32_t k;
    const uint32_t *orig_of, *orig_row_ptr;
    const uint32_t *comp;                // per cell: component of the light pairs' MST
    const uint32_t *hub;                 // the hub component
};

// The caller's index of arc x -> y (row x starts at rs, at cbase + rs in the
// caller's order).
__device__ __forceinline__ uint32_t caller_arc(const TreeScanArgs &a, uint32_t x, uint32_t rs,
                                               uint32_t cbase, uint32_t y) {
    const uint32_t want = caller_id(a.orig_of, y);
    uint32_t lo = rs, hi = a.row_ptr[x + 1];
    while (hi - lo > 1) {                // largest arc whose head is at or before y
        const uint32_t mid = lo + (hi - lo) / 2;
        if (caller_id(a.orig_of, a.adj[mid].x) <= want) lo = mid;
        else hi = mid;
    }
    return cbase + lo;
}

// Proposes bridge b over arc x -> y (x in the cell of smaller rank).  Weights
// of a narrow range make many bridges of a pair equal, and only the smallest
// arc counts: an arc of a later row is turned away before the search.
__device__ __forceinline__ void propose_bridge(const TreeScanArgs &a, uint32_t cx, uint32_t cy,
                                               uint64_t b, uint32_t x, uint32_t y) {
    auto *slot = reinterpret_cast<unsigned long long *>(&a.pairtab[pair_slot(cx, cy, a.k)]);
    unsigned long long cur = __ldg(slot);        // (a stale value is only larger)
    if (b < cur >> 32) cur = atomicMin(slot, (b << 32) | INF32);
    if (b > cur >> 32) return;
    const uint32_t rs = a.row_ptr[x], cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, x, rs);
    if (b == cur >> 32 && (uint32_t)cur < cbase + rs) return;    // a tie with an earlier row's arc
    atomicMin(slot, (b << 32) | caller_arc(a, x, rs, cbase, y));
}

// Arc `arc` = (v, head, w) of step 1, lu the head's label.
template <bool PAIRS>
__device__ __forceinline__ void tree_arc(const TreeScanArgs &a, uint32_t v, uint32_t lv,
                                         uint32_t arc, uint2 e, uint32_t lu) {
    if (lu == INF32) return;
    const uint64_t sum = ((uint64_t)e.y << a.lshift) + lu;       // the head's distance + w
    if (sum == lv) atomicMin(&a.pred_arc[v], arc);
    if (!PAIRS) return;
    const uint32_t mask = (1u << a.lshift) - 1u, cv = lv & mask, cu = lu & mask;
    if (cv >= cu) return;
    const uint64_t b = (lv >> a.lshift) + (sum >> a.lshift);
    if (b < a.delta) propose_bridge(a, cv, cu, b, v, e.x);
}

constexpr int TREE_ILP = 2;        // arcs in flight per lane (full occupancy matters more)

// PAIRS: step 1.  Else the predecessors of every vertex, for a Voronoi call:
// the rows of the vertices beyond delta too, whole.
template <bool PAIRS>
__global__ void __launch_bounds__(256, 8) tree_scan_kernel(const __grid_constant__ TreeScanArgs a) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_work = a.n_heavy_chunks + a.n_items;
    for (uint32_t wi = warp; wi < n_work; wi += nwarps) {
        if (wi < a.n_heavy_chunks) {
            const uint64_t item = a.heavy_chunks[wi];
            const uint32_t v = (uint32_t)(item >> 32), c = (uint32_t)item;
            const uint32_t lv = __ldg(&a.label32[v]);
            if (lv == INF32) continue;
            const bool far = lv >= a.near;           // the whole row, for the predecessor alone
            RowPiece p = row_piece(a.row_ptr[v], far ? a.row_ptr[v + 1] : a.lend[v], c * CHUNK, CHUNK);
            const uint2 *arcs = far ? a.adj : a.adj_w;
            for (; p.count; skip_arcs(p, 32 * TREE_ILP)) {
                uint2 x[TREE_ILP];
                uint32_t lu[TREE_ILP];
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q) {
                    x[q] = make_uint2(0, 0);                    // weight 0: no arc
                    if (32 * q + lane < p.count) x[q] = __ldcs(&arcs[p.first + 32 * q + lane]);
                }
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q) {
                    // (an arc heavier than the row's distance is not tight)
                    const bool look = x[q].y && ((PAIRS && !far) || x[q].y <= lv >> a.lshift);
                    lu[q] = look ? __ldg(&a.label32[x[q].x]) : INF32;
                }
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q)
                    tree_arc<PAIRS>(a, v, lv, p.first + 32 * q + lane, x[q], lu[q]);
            }
            continue;
        }
        const uint32_t v1 = __ldg(&a.items[wi - n_work + a.n_items + 1]);
        for (uint32_t vb = __ldg(&a.items[wi - n_work + a.n_items]); vb < v1; vb += 32) {
            const uint32_t v = vb + lane;
            uint32_t s = 0, deg = 0, lv = INF32;
            if (v < v1) {
                lv = __ldg(&a.label32[v]);
                if (lv < a.near || (!PAIRS && lv != INF32)) {
                    s = a.row_ptr[v];
                    const uint32_t r1 = a.row_ptr[v + 1];
                    deg = r1 - s >= HEAVY_DEG ? 0u : (lv < a.near ? a.lend[v] : r1) - s;
                }
            }
            const uint32_t rows = __ballot_sync(FULL, deg != 0);
            if (rows == 0) continue;
            const uint32_t incl = warp_inclusive_scan(deg);
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            const uint32_t excl = deg ? incl - deg : INF32;
            uint32_t before = 0;             // rows that start before the window
            for (uint32_t b = 0; b < total; b += 32 * TREE_ILP) {
                uint2 x[TREE_ILP];
                uint32_t lu[TREE_ILP], own[TREE_ILP], at[TREE_ILP], lo[TREE_ILP];
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q) {
                    const uint32_t w0 = b + 32 * q, j = w0 + lane;
                    const uint32_t starts = __reduce_or_sync(FULL, excl - w0 < 32 ? 1u << (excl - w0) : 0u);
                    own[q] = nth_set_bit(rows, before + (uint32_t)__popc(starts & (FULL >> (31 - lane))) - 1);
                    before += (uint32_t)__popc(starts);
                    at[q] = __shfl_sync(FULL, s - excl, own[q]) + j;
                    lo[q] = __shfl_sync(FULL, lv, own[q]);
                    x[q] = make_uint2(0, 0);
                    if (j < total) x[q] = __ldcs(&(PAIRS || lo[q] < a.near ? a.adj_w : a.adj)[at[q]]);
                }
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q) {
                    // (an arc heavier than the row's distance is not tight)
                    const bool look = x[q].y && (PAIRS || x[q].y <= lo[q] >> a.lshift);
                    lu[q] = look ? __ldg(&a.label32[x[q].x]) : INF32;
                }
#pragma unroll
                for (int q = 0; q < TREE_ILP; ++q)
                    tree_arc<PAIRS>(a, vb + own[q], lo[q], at[q], x[q], lu[q]);
            }
        }
    }
}

// Step 3: the rows of the vertices outside the hub component's cells.
__global__ void __launch_bounds__(256) rest_scan_kernel(const __grid_constant__ TreeScanArgs a) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_work = a.n_heavy_chunks + a.n_items;
    const uint32_t hub = *a.hub, mask = (1u << a.lshift) - 1u;
    // arc `at` of row v (the caller's index cbase + at)
    auto arc = [&](uint32_t v, uint32_t lv, uint32_t cc, uint32_t cbase, uint32_t at) {
        const uint2 e = __ldcs(&a.adj[at]);
        const uint32_t lu = __ldg(&a.label32[e.x]);
        const uint32_t cm = lu == INF32 ? cc : __ldg(&a.comp[lu & mask]);
        if (cm == cc) return;
        const uint32_t cv = lv & mask, cu = lu & mask;
        const uint64_t b = (uint64_t)(lv >> a.lshift) + e.y + (lu >> a.lshift);
        if (cv < cu) {
            auto *slot = reinterpret_cast<unsigned long long *>(&a.pairtab[pair_slot(cv, cu, a.k)]);
            const unsigned long long key = (b << 32) | (uint32_t)(cbase + at);
            if (key < __ldg(slot)) atomicMin(slot, key);
        } else if (cm == hub) {
            propose_bridge(a, cu, cv, b, e.x, v);    // the head's row is not read
        }
    };
    for (uint32_t wi = warp; wi < n_work; wi += nwarps) {
        if (wi < a.n_heavy_chunks) {
            const uint64_t item = a.heavy_chunks[wi];
            const uint32_t v = (uint32_t)(item >> 32), c = (uint32_t)item;
            const uint32_t lv = __ldg(&a.label32[v]);
            if (lv == INF32) continue;
            const uint32_t cc = __ldg(&a.comp[lv & mask]);
            if (cc == hub) continue;
            const uint32_t rs = a.row_ptr[v];
            const RowPiece p = row_piece(rs, a.row_ptr[v + 1], c * CHUNK, CHUNK);
            const uint32_t cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, v, rs);
            for (uint32_t j = lane; j < p.count; j += 32) arc(v, lv, cc, cbase, p.first + j);
            continue;
        }
        const uint32_t v1 = __ldg(&a.items[wi - n_work + a.n_items + 1]);
        for (uint32_t vb = __ldg(&a.items[wi - n_work + a.n_items]); vb < v1; vb += 32) {
            const uint32_t v = vb + lane;
            uint32_t s = 0, deg = 0, lv = INF32, cc = hub, cbase = 0;
            if (v < v1) {
                lv = __ldg(&a.label32[v]);
                if (lv != INF32) cc = __ldg(&a.comp[lv & mask]);
                if (cc != hub) {
                    s = a.row_ptr[v];
                    deg = a.row_ptr[v + 1] - s;
                    if (deg >= HEAVY_DEG) deg = 0;   // covered by the chunk list
                    if (deg) cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, v, s);
                }
            }
            if (!__any_sync(FULL, deg)) continue;
            const uint32_t incl = warp_inclusive_scan(deg);
            const uint32_t excl = incl - deg;
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            for (uint32_t b = 0; b < total; b += 32) {
                const uint32_t j = b + lane;
                const uint32_t own = warp_owner_search(excl, j < total ? j : 0);
                const uint32_t at = __shfl_sync(FULL, s - excl, own) + j;
                const uint32_t lo = __shfl_sync(FULL, lv, own), co = __shfl_sync(FULL, cc, own);
                const uint32_t bo = __shfl_sync(FULL, cbase, own);
                if (j < total) arc(vb + own, lo, co, bo, at);
            }
        }
    }
}

// Arcs per component, by a sample of arcs spread over all of them.
constexpr uint32_t HUB_SAMPLES = 1u << 15;
__global__ void hub_sample_kernel(const __grid_constant__ TreeScanArgs a, uint32_t n, uint64_t m,
                                  uint32_t *count) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= HUB_SAMPLES) return;
    const uint32_t arc = (uint32_t)(m * i / HUB_SAMPLES);
    uint32_t lo = 0, hi = n;             // largest v with row_ptr[v] <= arc
    while (hi - lo > 1) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (a.row_ptr[mid] <= arc) lo = mid;
        else hi = mid;
    }
    const uint32_t lv = a.label32[lo];
    if (lv != INF32) atomicAdd(&count[a.comp[lv & ((1u << a.lshift) - 1u)]], 1u);
}

// The component with the largest count (one block).
__global__ void __launch_bounds__(1024) hub_pick_kernel(const uint32_t *count, uint32_t k, uint32_t *hub) {
    __shared__ unsigned long long best;
    if (threadIdx.x == 0) best = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (uint32_t c = threadIdx.x; c < k; c += blockDim.x) {
        const unsigned long long x = ((unsigned long long)count[c] << 32) | c;
        if (x > mine) mine = x;
    }
    atomicMax(&best, mine);
    __syncthreads();
    if (threadIdx.x == 0) *hub = (uint32_t)best;
}

// ---------------------------------------------------------------------------
// ordered compaction of the pair table: entries != INF in slot order,
// i.e. ascending (rank a, rank b)
// ---------------------------------------------------------------------------

constexpr uint32_t CT_THREADS = 256;
constexpr uint32_t CT_PER_THREAD = 8;
constexpr uint32_t CT_TILE = CT_THREADS * CT_PER_THREAD;

__global__ void __launch_bounds__(CT_THREADS) pair_count_kernel(const uint64_t *__restrict__ tab,
                                                                uint64_t slots,
                                                                uint32_t *__restrict__ tile_cnt) {
    __shared__ uint32_t wsum[CT_THREADS / 32];
    uint64_t base = (uint64_t)blockIdx.x * CT_TILE + (uint64_t)threadIdx.x * CT_PER_THREAD;
    uint32_t c = 0;
#pragma unroll
    for (uint32_t i = 0; i < CT_PER_THREAD; ++i)
        if (base + i < slots && tab[base + i] != INF64) ++c;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if (lane_id() == 0) wsum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (uint32_t w = 0; w < CT_THREADS / 32; ++w) t += wsum[w];
        tile_cnt[blockIdx.x] = t;
    }
}

// single block: exclusive scan of the tile counts, total into *n_pairs
__global__ void __launch_bounds__(1024) tile_scan_kernel(uint32_t *tile_cnt, uint32_t n_tiles,
                                                         uint32_t *n_pairs) {
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < n_tiles; base += blockDim.x) {
        uint32_t i = base + threadIdx.x;
        uint32_t x = i < n_tiles ? tile_cnt[i] : 0;
        uint32_t incl = warp_inclusive_scan(x);
        if (lane_id() == 31) wsum[threadIdx.x >> 5] = incl;
        __syncthreads();
        if (threadIdx.x < 32) {
            uint32_t ws = wsum[threadIdx.x];
            uint32_t wi = warp_inclusive_scan(ws);
            wsum[threadIdx.x] = wi - ws;
        }
        __syncthreads();
        uint32_t excl = carry + wsum[threadIdx.x >> 5] + incl - x;
        if (i < n_tiles) tile_cnt[i] = excl;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = excl + x;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_pairs = carry;
}

__global__ void __launch_bounds__(CT_THREADS) pair_write_kernel(
    const uint64_t *__restrict__ tab, uint64_t slots, uint32_t k,
    const uint32_t *__restrict__ tile_off, uint64_t *e_key, uint32_t *e_ra, uint32_t *e_rb,
    uint32_t *e_arc, uint32_t *e_mst) {
    __shared__ uint32_t wsum[CT_THREADS / 32];
    uint64_t base = (uint64_t)blockIdx.x * CT_TILE + (uint64_t)threadIdx.x * CT_PER_THREAD;
    uint64_t vals[CT_PER_THREAD];
    uint32_t c = 0;
#pragma unroll
    for (uint32_t i = 0; i < CT_PER_THREAD; ++i) {
        vals[i] = base + i < slots ? tab[base + i] : INF64;
        if (vals[i] != INF64) ++c;
    }
    uint32_t incl = warp_inclusive_scan(c);
    if (lane_id() == 31) wsum[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t ws = threadIdx.x < CT_THREADS / 32 ? wsum[threadIdx.x] : 0;
        uint32_t wi = warp_inclusive_scan(ws);
        if (threadIdx.x < CT_THREADS / 32) wsum[threadIdx.x] = wi - ws;
    }
    __syncthreads();
    uint32_t out = tile_off[blockIdx.x] + wsum[threadIdx.x >> 5] + incl - c;
#pragma unroll
    for (uint32_t i = 0; i < CT_PER_THREAD; ++i) {
        if (vals[i] == INF64) continue;
        uint64_t slot = base + i;
        uint32_t ra, rb;
        slot_to_pair(slot, k, ra, rb);
        e_key[out] = (vals[i] & 0xFFFFFFFF00000000ull) | slot;    // (b << 32) | slot
        e_ra[out] = ra;
        e_rb[out] = rb;
        e_arc[out] = (uint32_t)vals[i];
        e_mst[out] = 0;
        ++out;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t launch_scan(const DevGraph &g, Workspace &ws, uint32_t k, bool pairs,
                        cudaStream_t s) {
    ScanArgs a;
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.heavy_chunks = g.heavy_chunks;
    a.n_heavy_chunks = g.n_heavy_chunks;
    a.n = g.n;
    a.label = ws.label;
    a.label32 = ws.label32;
    a.lshift = ws.lshift;
    a.pred_arc = ws.pred_arc;
    a.pairtab = ws.pairtab;
    a.k = k;
    a.pairs = pairs && k > 1;
    a.err = &ws.ctl->err;
    a.orig_of = g.orig_of;
    a.orig_row_ptr = g.orig_row_ptr;
    if (a.pairs) {
        uint64_t slots = (uint64_t)k * (k - 1) / 2;
        cudaError_t e = cudaMemsetAsync(ws.pairtab, 0xFF, slots * sizeof(uint64_t), s);
        if (e != cudaSuccess) return e;
    }
    const uint64_t cap = (uint64_t)current_sm_count() * 32;
    // hub chunks in pieces while they leave most of the grid's warps idle
    a.subs = g.n_heavy_chunks * (uint64_t)SCAN_SUBS <= cap * 8 ? SCAN_SUBS : 1u;
    a.items = g.scan_items();
    a.n_items = g.n_scan_items();
    uint64_t work = (uint64_t)g.n_heavy_chunks * a.subs + g.n_scan_items();
    uint64_t blocks = (work + 7) / 8;          // 8 warps per block
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    if (ws.narrow) scan_kernel<true><<<(unsigned)blocks, 256, 0, s>>>(a);
    else scan_kernel<false><<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_compact_pairs(Workspace &ws, uint32_t k, cudaStream_t s) {
    uint64_t slots = k > 1 ? (uint64_t)k * (k - 1) / 2 : 0;
    if (slots == 0) return cudaMemsetAsync(&ws.ctl->n_pairs, 0, sizeof(uint32_t), s);
    uint32_t tiles = (uint32_t)((slots + CT_TILE - 1) / CT_TILE);
    pair_count_kernel<<<tiles, CT_THREADS, 0, s>>>(ws.pairtab, slots, ws.tile_off);
    tile_scan_kernel<<<1, 1024, 0, s>>>(ws.tile_off, tiles, &ws.ctl->n_pairs);
    pair_write_kernel<<<tiles, CT_THREADS, 0, s>>>(ws.pairtab, slots, k, ws.tile_off, ws.e_key,
                                                   ws.e_ra, ws.e_rb, ws.e_arc, ws.e_mst);
    return cudaGetLastError();
}

// The tree-only scan serves a query whose label width and weights make it
// exact (narrow labels of two rank bits or more cannot overflow a bridge), with
// rows split by weight, where it pays.
bool tree_scan_applies(const DevGraph &g, const Workspace &ws, uint32_t k, uint32_t delta) {
    const bool exact = ws.narrow && ws.lshift >= 2 && g.max_w < 0x80000000u &&
                       active_lend(g, delta) && k > 1 && !small_tail(k);
    if (g.tree_scan >= 0) return exact && g.tree_scan;
    return exact && tree_scan_pays(g.m, k, delta, g.max_w);
}

static TreeScanArgs tree_scan_args(const DevGraph &g, const Workspace &ws, uint32_t k, uint32_t delta) {
    TreeScanArgs a;
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.adj_w = g.adj_w;
    a.lend = g.lend;
    a.heavy_chunks = g.heavy_chunks;
    a.n_heavy_chunks = g.n_heavy_chunks;
    a.items = g.scan_items();
    a.n_items = g.n_scan_items();
    a.delta = delta;
    a.near = near_label(ws, delta);
    a.label32 = ws.label32;
    a.lshift = ws.lshift;
    a.pred_arc = ws.pred_arc;
    a.pairtab = ws.pairtab;
    a.k = k;
    a.orig_of = g.orig_of;
    a.orig_row_ptr = g.orig_row_ptr;
    a.comp = ws.comp;
    a.hub = ws.hub;
    return a;
}

cudaError_t launch_tree_scan(const DevGraph &g, Workspace &ws, uint32_t k, uint32_t delta,
                             const Geometry &geo, cudaStream_t s) {
    const TreeScanArgs a = tree_scan_args(g, ws, k, delta);
    const uint64_t slots = (uint64_t)k * (k - 1) / 2;
    cudaError_t e = cudaMemsetAsync(ws.pairtab, 0xFF, slots * sizeof(uint64_t), s);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)current_sm_count() * 32;
    tree_scan_kernel<true><<<blocks, 256, 0, s>>>(a);
    e = launch_compact_pairs(ws, k, s);
    if (e == cudaSuccess) e = launch_mst(ws, k, geo, (uint64_t)delta << 32, s);
    // (the MST is done with its hooks: they count the samples)
    if (e == cudaSuccess) e = cudaMemsetAsync(ws.hook, 0, (size_t)k * 4, s);
    if (e != cudaSuccess) return e;
    hub_sample_kernel<<<HUB_SAMPLES / 256, 256, 0, s>>>(a, g.n, g.m, ws.hook);
    hub_pick_kernel<<<1, 1024, 0, s>>>(ws.hook, k, ws.hub);
    rest_scan_kernel<<<blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// Predecessors alone, by the light part of most rows (R-MAT 22, weights to
// 10^5, k = 64: Voronoi call 1.62 ms, with the full scan 1.82).  It sees no
// overflow.  A distance that does not fit a narrow label is found while it is
// relaxed, but the relaxation leaves out arcs of weight 2^32 - 1: with one in
// the graph the full scan looks for reached vertices next to unreached ones.
bool pred_scan_applies(const DevGraph &g, const Workspace &ws, uint32_t delta) {
    return ws.narrow && active_lend(g, delta) && g.max_w < INF32;
}

cudaError_t launch_pred_scan(const DevGraph &g, Workspace &ws, uint32_t k, uint32_t delta,
                             cudaStream_t s) {
    const TreeScanArgs a = tree_scan_args(g, ws, k, delta);
    const uint64_t work = (uint64_t)g.n_heavy_chunks + g.n_scan_items();
    const uint64_t blocks = std::min<uint64_t>((work + 7) / 8, (uint64_t)current_sm_count() * 32);
    tree_scan_kernel<false><<<(unsigned)std::max<uint64_t>(blocks, 1), 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace stn
