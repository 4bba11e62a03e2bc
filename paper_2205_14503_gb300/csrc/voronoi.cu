// Voronoi cells of all seeds at once (Algorithm 2 Step 1; Algorithm 4 is the
// paper's asynchronous vertex-centric form of the same fixed point).
//
// Every vertex v holds one packed label (d1(src(v), v) << 32) | rank(src(v)).
// Relaxing an arc u -> v proposes (d(u) + d(u,v)) << 32 | rank(u) and keeps
// the minimum with a 64-bit atomicMin, so the fixed point is, per vertex,
// the lexicographic minimum over seeds of (distance, seed rank): the
// nearest seed, ties to the smallest seed id.  The fixed point does not
// depend on the order in which relaxations land.
//
// Order of work: a near/far frontier (a two-bucket delta-stepping).  The
// paper prioritises low-distance messages in its message queue (Section
// "Distributed Implementation"); on the GPU the same effect comes from
// relaxing only vertices whose distance is below a threshold T (near) and
// parking the rest (far) until the near frontier drains, then raising T by
// delta.  One persistent cooperative kernel runs all iterations with a
// bounded grid barrier between them.
//
// Light and heavy arcs (the edge classes of delta-stepping): while a band
// [T - delta, T) iterates, only arcs lighter than delta are relaxed, since
// a heavier arc out of the band cannot land inside it.  Every vertex
// relaxed in the band is listed once; when the band's frontier drains, one
// extra pass relaxes the heavy arcs of the listed vertices with their final
// labels, so a vertex improved several times inside its band (a hub reached
// by many light paths) scans its heavy arcs once.  All of its proposals land
// at or above T, in the far pile.  The split is on only when some arc
// weight reaches delta.
//
// Pull form of the heavy-arc pass (with the far scan): once a band has
// drained, every label below T is final, and a heavy proposal can only
// change a vertex still at or above T.  So instead of pushing the heavy
// arcs of the band's vertices, every unsettled vertex may read its own
// heavy arcs and the labels at their other ends, keeping the best proposal
// from those below T.  Both forms reach the same labels; the pass takes
// the form that reads fewer arcs.  On a small-world graph the first band
// holds most of the vertices and nearly all heavy arcs, while the vertices
// left unsettled have few (direction-optimising search, Beamer et al.,
// applied to delta-stepping's heavy-arc phase).
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace stn {

struct SsspArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;
    uint32_t n;
    uint64_t *label;         // 64-bit labels (the wide kernel)
    uint32_t *label32;       // narrow labels (the narrow kernel)
    uint32_t lshift;         // rank bits of a narrow label
    uint32_t lstep;          // 1 << lshift: a narrow label's step per unit of distance
    uint64_t lmiss;          // sums of label and step at or above this do not fit
    uint32_t *stamp_near;
    uint32_t *stamp_far;
    uint32_t *q0, *q1;
    uint64_t *hq0, *hq1;
    uint32_t *far0, *far1;
    Control *ctl;
    uint32_t delta;
    uint32_t max_iters;
    uint32_t base_near;
    uint32_t base_far;
    uint32_t heavy_cap;
    uint32_t local_rounds;   // warp-local relaxation rounds per iteration (0 = off)
    uint32_t *stamp_band;    // band-list membership tags
    uint32_t *band_q;        // vertices relaxed in the current band
    uint64_t *band_hq;       // heavy-row chunks of listed high-degree vertices
    uint32_t base_band;
    uint32_t defer;          // light/heavy arc split on
    uint32_t trace;          // record per-iteration relaxation counts
    // Dense frontiers (with the far scan, without local rounds): a large
    // frontier is a bitmap (one bit per vertex, set with a fire-and-forget
    // atomicOr) read in id order by the next iteration, and the band list
    // of the light/heavy split is a bitmap too; hubs keep their chunk
    // queues.  Ids below n_big may have HEAVY_DEG arcs or more, ids at or
    // above it have fewer (the degree order makes this a bound).
    uint32_t dense;
    uint32_t pull;           // heavy-arc passes: 0 push, 1 by cost, 2 pull
    uint32_t step0;          // first threshold inside the first band (0: the band)
    uint32_t thin;           // far pile: a frontier below this size splits the pile early
    uint32_t thin_rounds;    // ... and takes this many warp-local rounds
    uint32_t tail;           // 1: after a pull pass the rest runs as one unbounded band
    uint64_t m;              // arcs (the first bound on a pull pass's cost)
    uint32_t n_big;
    uint32_t n_live;         // ids at or above it have no arcs
    uint32_t n_words;        // bitmap words, ceil(n / 32)
    uint32_t *nbm0, *nbm1;   // near bitmaps, alternating by iteration
    uint32_t *bbm;           // band bitmap
    // vertex ranges that dense iterations hand to the warps (n_items of
    // them), and the coarser ones for a sparse bitmap
    const uint32_t *__restrict__ items;
    const uint32_t *__restrict__ sparse_items;
    uint32_t n_items, n_sparse_items;
    // with the split: end of each row's light part in the weight-partitioned
    // adjacency `adj` (null: rows are unpartitioned and arcs are filtered)
    const uint32_t *lend;
};

// ---------------------------------------------------------------------------
// init (Algorithm 3, INITIALIZATION): every label at infinity, then each
// seed at distance 0 in its own cell and on the first frontier.
// ---------------------------------------------------------------------------

__global__ void init_labels_kernel(uint32_t n, uint64_t *__restrict__ label,
                                   uint32_t *__restrict__ label32,
                                   uint32_t *__restrict__ pred_arc) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (label32) label32[v] = INF32;
        else label[v] = INF64;
        pred_arc[v] = INF32;
    }
}

__global__ void init_seeds_kernel(const uint32_t *__restrict__ row_ptr,
                                  const uint32_t *__restrict__ lend, const int32_t *seeds,
                                  const uint32_t *__restrict__ new_of,
                                  uint32_t k, uint64_t *label, uint32_t *label32,
                                  uint32_t *pred_arc,
                                  uint32_t *stamp_near, uint32_t tag0, uint32_t *q0,
                                  uint64_t *hq0, uint32_t heavy_cap, uint32_t n, Control *ctl) {
    uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r == 0) {
        ctl->far_min[0] = INF32;
        ctl->far_min[1] = INF32;
        ctl->far_min[2] = INF32;
    }
    if (r >= k) return;
    uint32_t s = internal_id(new_of, (uint32_t)seeds[r]);
    if (label32) label32[s] = r;          // distance 0, cell = rank r
    else label[s] = (uint64_t)r;
    pred_arc[s] = SEED_ARC;
    stamp_near[s] = tag0;
    uint32_t rs = row_ptr[s], deg = (lend ? lend[s] : row_ptr[s + 1]) - rs;   // near part
    if (deg >= HEAVY_DEG) {
        uint32_t nc = (deg + CHUNK - 1) / CHUNK;
        uint32_t base = atomicAdd(&ctl->heavy_count[0], nc);
        if (base + nc > heavy_cap) { atomicOr(&ctl->err, ERR_CAPACITY); return; }
        for (uint32_t c = 0; c < nc; ++c) hq0[base + c] = ((uint64_t)s << 32) | c;
    } else {
        uint32_t slot = atomicAdd(&ctl->near_count[0], 1u);
        if (slot >= n) { atomicOr(&ctl->err, ERR_CAPACITY); return; }
        q0[slot] = s;
    }
}

// ---------------------------------------------------------------------------
// relaxation: U arcs in flight per lane; frontier appends staged per block
// ---------------------------------------------------------------------------

constexpr int ILP = 4;                 // arcs per lane per round group (relax_group's
                                       // early exit tests imp[0..3] by name: keep 4)
constexpr uint32_t NEAR_STAGE = 4096;  // block staging capacity (near items)
constexpr uint32_t SSSP_WARPS = 8;     // warps per block (256 threads)
constexpr uint32_t NEAR_REGION = NEAR_STAGE / SSSP_WARPS;   // one region per warp
constexpr uint32_t FAR_STAGE = 1024;   // block staging capacity (far items)
constexpr uint32_t BAND_STAGE = 2048;  // block staging capacity (band-list items)
constexpr uint32_t BAND_REGION = BAND_STAGE / SSSP_WARPS;
constexpr int SPLIT_ILP = 4;           // 32-vertex chunks per warp step in a band split
constexpr uint32_t SUB_CHUNKS = 4;     // pieces of a hub chunk while hub chunks are few
static_assert(CHUNK / SUB_CHUNKS >= 32 * ILP, "a piece is at least one relax_group");
constexpr int PULL_ILP = 4;            // 32-vertex chunks per warp step in a pull pass

// Where the appends of one processing segment go.
struct PushTargets {
    uint32_t *qn;        // light queue of the next iteration
    uint32_t *qn_count;
    uint64_t *hqn;       // heavy-chunk queue of the next iteration
    uint32_t *hqn_count;
    uint32_t *farq;      // far pile of the current phase
    uint32_t *far_count;
    uint32_t *far_min;
    uint32_t *bandq;     // band list and its fill counter
    uint32_t *band_count;
    uint32_t tag_next;
    uint32_t tag_far;
    uint64_t Tl;         // the threshold as a label of the kernel's width
    // Near pushes of light vertices set bits of nbm (the next iteration
    // reads the bitmap) instead of going through the queue.
    bool dense;
    uint32_t *nbm;
    // With warp-local rounds: every improvement appends its vertex to the
    // improving warp's region with no stamp (a region may hold a vertex
    // twice, and a warp-local round simply reads the current label); the
    // near stamps deduplicate items only on their way to the global queue.
    bool nostamp;
    uint32_t *nostamp_stamp;     // the near stamps (for the deduplication)
    unsigned long long *hsum;    // receives the warps' heavy-arc sums (null: none)
    // end of each row's part relaxed by a near vertex (the light part while
    // the light/heavy split is on); null: whole rows
    const uint32_t *lend;
};

// Per-block staging buffers.  Near and band-list appends go to one region
// per warp, which only that warp touches: a full region moves to the global
// queue with one global atomicAdd (one per region, not one per append: a
// single queue counter that every warp bumps on every append serialises the
// whole grid on one L2 address), and the rest moves at the end of the
// segment (flush_stage).  In the local rounds a warp relaxes its own near
// region.  Far appends share one block buffer (shared-memory atomics).
struct Stage {
    uint32_t near_buf[NEAR_STAGE];
    uint32_t far_buf[FAR_STAGE];
    uint32_t band_buf[BAND_STAGE];
    uint32_t band_n[SSSP_WARPS];    // items staged per band region
    uint32_t dn_near[SSSP_WARPS];   // bits set in the near bitmap by each warp
    uint32_t dn_band[SSSP_WARPS];   // bits set in the band bitmap by each warp
    uint32_t hs[SSSP_WARPS];        // heavy arcs listed (or pulled) by each warp
    uint32_t near_n[SSSP_WARPS];    // items staged per warp region
    uint32_t local_lo[SSSP_WARPS];  // region[0, local_lo) was relaxed by its warp already
    uint32_t near_off[SSSP_WARPS];  // flush: offset of each region's rest
    uint32_t far_n, far_min;
    uint32_t base_near, base_far;
};

__device__ __forceinline__ void stage_reset(Stage &st) {
    if (threadIdx.x == 0) {
        st.far_n = 0;
        st.far_min = INF32;
    }
    if (threadIdx.x < SSSP_WARPS) {
        st.near_n[threadIdx.x] = 0;
        st.band_n[threadIdx.x] = 0;
        st.dn_near[threadIdx.x] = 0;
        st.dn_band[threadIdx.x] = 0;
        st.hs[threadIdx.x] = 0;
        st.local_lo[threadIdx.x] = 0;
    }
    __syncthreads();
}

// Moves the block's staged appends to the global queues.  Called by all
// threads of the block; ends with the staging buffers still holding data
// (stage_reset clears them at the next segment).
__device__ __forceinline__ void flush_stage(Stage &st, const PushTargets &t, uint32_t n,
                                            uint32_t *err) {
    __syncthreads();
    const uint32_t nf = min(st.far_n, FAR_STAGE);
    if (threadIdx.x < 32) {
        // lane w < SSSP_WARPS sums up warp w's region; the atomics whose
        // results are needed go out together, from different lanes
        const uint32_t w = threadIdx.x;
        uint32_t nn = 0, dnn = 0, dnb = 0, hs = 0;
        if (w < SSSP_WARPS) {
            const uint32_t hi = min(st.near_n[w], NEAR_REGION), lo = st.local_lo[w];
            nn = !t.nostamp && hi > lo ? hi - lo : 0;
            // bits set in the bitmaps count as items (a vertex set twice
            // counts twice): the counts only size the next iteration and
            // show that a frontier or band list is non-empty
            dnn = st.dn_near[w];
            dnb = st.dn_band[w];
            hs = st.hs[w];
        }
        const uint32_t incl = warp_inclusive_scan(nn);
        if (w < SSSP_WARPS) st.near_off[w] = incl - nn;
        nn = __shfl_sync(FULL, incl, 31);
        dnn = __reduce_add_sync(FULL, dnn);
        dnb = __reduce_add_sync(FULL, dnb);
        unsigned long long hsum = hs;
        if (t.hsum) {
#pragma unroll
            for (int o = SSSP_WARPS / 2; o >= 1; o >>= 1) hsum += __shfl_xor_sync(FULL, hsum, o);
        }
        if (w == 0) {
            if (dnn) atomicAdd(t.qn_count, dnn);
            if (dnb) atomicAdd(t.band_count, dnb);
            if (t.hsum && hsum) atomicAdd(t.hsum, hsum);
            if (st.far_min != INF32) atomicMin(t.far_min, st.far_min);
            st.base_near = nn ? atomicAdd(t.qn_count, nn) : 0;
        } else if (w == 1) {
            st.base_far = nf ? atomicAdd(t.far_count, nf) : 0;
        }
    }
    __syncthreads();
    {   // each warp moves the rest of its own regions
        const uint32_t w = threadIdx.x >> 5;
        const uint32_t hi = min(st.near_n[w], NEAR_REGION), lo = st.local_lo[w];
        if (t.nostamp) {            // deduplicated on the way
            for (uint32_t i0 = lo; i0 < hi; i0 += 32) {
                const uint32_t i = i0 + lane_id();
                queue_append(i < hi, i < hi ? st.near_buf[w * NEAR_REGION + i] : 0u, t.qn,
                             t.qn_count, n, err, t.nostamp_stamp, t.tag_next);
            }
        } else {
            for (uint32_t i = lo + lane_id(); i < hi; i += 32) {
                uint32_t slot = st.base_near + st.near_off[w] + (i - lo);
                if (slot < n) t.qn[slot] = st.near_buf[w * NEAR_REGION + i];
                else atomicOr(err, ERR_CAPACITY);
            }
        }
        const uint32_t nb = min(st.band_n[w], BAND_REGION);
        if (nb) {
            uint32_t base = 0;
            if (lane_id() == 0) base = atomicAdd(t.band_count, nb);
            base = __shfl_sync(FULL, base, 0);
            for (uint32_t i = lane_id(); i < nb; i += 32) {
                if (base + i < n) t.bandq[base + i] = st.band_buf[w * BAND_REGION + i];
                else atomicOr(err, ERR_CAPACITY);
            }
        }
    }
    for (uint32_t i = threadIdx.x; i < nf; i += blockDim.x) {
        uint32_t slot = st.base_far + i;
        if (slot < n) t.farq[slot] = st.far_buf[i];
        else atomicOr(err, ERR_CAPACITY);
    }
}

// Near appends of N vertices per lane: high-degree vertices become CHUNK-arc
// items of the heavy queue (one atomicAdd for the warp's), the rest go
// through the staging buffer.  `flush`: a full warp region may move to the
// global queue (not during the warp-local rounds, which index into it).
template <int N>
__device__ __forceinline__ void push_near(const SsspArgs &a, Stage &st, const PushTargets &t,
                                          bool flush, const bool (&want)[N],
                                          const uint32_t (&v)[N], const uint32_t (&deg)[N]) {
    bool light[N];
    uint32_t nc = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        light[i] = want[i] && deg[i] < HEAVY_DEG;
        if (want[i] && !light[i]) nc += (deg[i] + CHUNK - 1) / CHUNK;
    }
    const uint32_t w = threadIdx.x >> 5;
    region_append_n<N>(light, v, st.near_buf + w * NEAR_REGION, &st.near_n[w], NEAR_REGION,
                       flush, t.qn, t.qn_count, a.n, &a.ctl->err,
                       t.nostamp ? a.stamp_near : nullptr, t.tag_next);
    if (!__any_sync(FULL, nc)) return;
    const uint32_t incl = warp_inclusive_scan(nc);
    uint32_t at = 0;
    if (lane_id() == 31) at = atomicAdd(t.hqn_count, incl);
    at = __shfl_sync(FULL, at, 31);
    if (at + __shfl_sync(FULL, incl, 31) > a.heavy_cap) {
        if (lane_id() == 0) atomicOr(&a.ctl->err, ERR_CAPACITY);
        return;
    }
    at += incl - nc;
    // the chunk lists, one hub after another: the whole warp writes each
#pragma unroll
    for (int i = 0; i < N; ++i)
        for (uint32_t m = __ballot_sync(FULL, want[i] && !light[i]); m; m &= m - 1) {
            const uint32_t l = __ffs(m) - 1;
            const uint32_t vl = __shfl_sync(FULL, v[i], l), base = __shfl_sync(FULL, at, l);
            const uint32_t n = (__shfl_sync(FULL, deg[i], l) + CHUNK - 1) / CHUNK;
            for (uint32_t c = lane_id(); c < n; c += 32) t.hqn[base + c] = ((uint64_t)vl << 32) | c;
            if (lane_id() == l) at += n;
        }
}

// Far appends of N vertices per lane: want[i] appends v[i] to the pile
// (first time this phase); cand[i] marks every far proposal, so far_min
// bounds the pile from below even for vertices already in it.
template <bool SCAN, int N, class Dist>
__device__ __forceinline__ void push_far(const SsspArgs &a, Stage &st, const PushTargets &t,
                                         const bool (&want)[N], const bool (&cand)[N],
                                         const uint32_t (&v)[N], Dist dist) {
    uint32_t m = INF32;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (cand[i]) m = min(m, dist(i));
    m = __reduce_min_sync(FULL, m);
    if (m == INF32) return;              // nothing far
    if (lane_id() == 0) atomicMin(&st.far_min, m);
    if constexpr (!SCAN) {               // (no pile with the scan)
        // one claim of the block's buffer for the warp's appends; what does
        // not fit goes to the pile
        uint32_t mask[N], k = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            mask[i] = __ballot_sync(FULL, want[i]);
            k += (uint32_t)__popc(mask[i]);
        }
        if (k == 0) return;
        uint32_t at = 0;
        if (lane_id() == 0) at = atomicAdd(&st.far_n, k);
        at = __shfl_sync(FULL, at, 0);
        const bool fits = at + k <= FAR_STAGE;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t slot = at + (uint32_t)__popc(mask[i] & lanemask_lt());
            if (want[i] && slot < FAR_STAGE) st.far_buf[slot] = v[i];
            if (!fits) {
                const uint32_t g = warp_append(want[i] && slot >= FAR_STAGE, t.far_count, a.n,
                                               &a.ctl->err);
                if (g != INF32) t.farq[g] = v[i];
            }
            at += (uint32_t)__popc(mask[i]);
        }
    }
}

// Label of v in the 64-bit form (read past L1: other blocks write it).
template <bool NARROW>
__device__ __forceinline__ uint64_t sssp_label(const SsspArgs &a, uint32_t v) {
    if (NARROW) return widen_label(ldcg_u32(&a.label32[v]), a.lshift);
    return ldcg_u64(&a.label[v]);
}

// Labels in the width of the kernel: the hot relaxation compares and sends
// them as stored.  A narrow proposal is one multiply-add, lab + (w << shift)
// in 64 bits, whose order and overflow tell everything; widening every
// label to 64 bits cost twice the instructions.
template <bool NARROW>
struct LabelOf {
    using T = uint64_t;
};
template <>
struct LabelOf<true> {
    using T = uint32_t;
};

template <bool NARROW>
__device__ __forceinline__ typename LabelOf<NARROW>::T raw_label(const SsspArgs &a, uint32_t v) {
    if constexpr (NARROW) return ldcg_u32(&a.label32[v]);
    else return ldcg_u64(&a.label[v]);
}

// The smallest label of a distance at or above T (saturating: with the far
// side empty every label is below it but the unreached one).
template <bool NARROW>
__device__ __forceinline__ uint64_t threshold_label(const SsspArgs &a, uint64_t T) {
    if (NARROW) return T >= (1ull << (32 - a.lshift)) ? INF32 : T << a.lshift;
    return T >= INF32 ? INF64 : T << 32;
}

// One group of up to N arcs per lane: the arc records and their tails'
// labels (`valid`: this lane has arc u).
template <bool NARROW, int N>
struct ArcGroup {
    uint2 e[N];
    typename LabelOf<NARROW>::T lab[N];
    bool valid[N];
};

// Relaxes a group's arcs of weight in [wlo, whi).  The loads and atomics of
// the N arcs are issued back to back so their latencies overlap.
// With `precheck` a plain load of the head's label comes first and only
// improving proposals issue the atomic: right for thick frontiers, where
// L2 atomic throughput is the limit; thin frontiers are latency-bound and
// skip the extra dependent load.
// NARROW kernels flag (narrow_miss) any proposal whose distance does not fit
// a 32-bit label, which the host answers with a 64-bit rerun.
template <bool NARROW, bool SCAN, int N>
__device__ __forceinline__ void relax_group(const SsspArgs &a, Stage &st, const PushTargets &t,
                                            const ArcGroup<NARROW, N> &g, bool flush, bool precheck, uint32_t wlo,
                                            uint32_t whi, uint32_t &attempts,
                                            uint32_t &improved, bool &narrow_miss) {
    using L = typename LabelOf<NARROW>::T;
    L nl[N], cur[N];
    bool want[N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
        want[u] = g.valid[u] && g.e[u].y >= wlo && g.e[u].y < whi;
        attempts += want[u];
        cur[u] = (L)~0ull;
        if constexpr (NARROW) {
            const uint64_t sum = (uint64_t)g.e[u].y * a.lstep + g.lab[u];
            if (want[u] && sum >= a.lmiss) {
                narrow_miss = true;
                want[u] = false;
            }
            nl[u] = (uint32_t)sum;
        } else {
            // proposals at or above 2^32 - 1 are skipped; the scan reports the overflow
            const uint64_t nd = (g.lab[u] >> 32) + (uint64_t)g.e[u].y;
            want[u] = want[u] && nd < INF32;
            nl[u] = (nd << 32) | (g.lab[u] & 0xFFFFFFFFull);
        }
        if (precheck && want[u]) cur[u] = raw_label<NARROW>(a, g.e[u].x);
    }
    bool imp[N], fr[N];
    bool any = false;
#pragma unroll
    for (int u = 0; u < N; ++u) {
        imp[u] = fr[u] = false;
        if (want[u] && nl[u] < cur[u]) {
            const bool far = SCAN && nl[u] >= (L)t.Tl;
            if constexpr (NARROW) {
                // a far proposal needs no answer (nothing is queued for it):
                // a fire-and-forget reduction
                if (far) atomicMin(&a.label32[g.e[u].x], nl[u]);
                else imp[u] = nl[u] < atomicMin(&a.label32[g.e[u].x], nl[u]);
            } else {
                auto *dst = reinterpret_cast<unsigned long long *>(&a.label[g.e[u].x]);
                if (far) atomicMin(dst, (unsigned long long)nl[u]);
                else imp[u] = nl[u] < atomicMin(dst, (unsigned long long)nl[u]);
            }
            fr[u] = far;
        }
        any |= imp[u] | fr[u];
    }
    // rounds that improve nothing skip the append machinery
    if (!__any_sync(FULL, any)) return;
    bool to_near[N], to_far[N], cand[N];
    uint32_t deg[N], vs[N];
    uint32_t dn = 0;
#pragma unroll
    for (int u = 0; u < N; ++u) {
        to_near[u] = to_far[u] = false;
        cand[u] = fr[u];         // a fire-and-forget far proposal still bounds far_min
        deg[u] = 0;
        const uint32_t v = vs[u] = g.e[u].x;
        if (!imp[u]) continue;
        ++improved;
        if (SCAN && nl[u] < (L)t.Tl && t.dense) {
            // a light vertex sets its bit; a possible hub (id below n_big)
            // reads its degree first and, if it is one, joins the chunk queue
            if (v < a.n_big) {
                const uint32_t r0 = a.row_ptr[v];
                deg[u] = (t.lend ? t.lend[v] : a.row_ptr[v + 1]) - r0;
            }
            if (deg[u] >= HEAVY_DEG) {
                to_near[u] = atomicExch(&a.stamp_near[v], t.tag_next) != t.tag_next;
            } else {
                atomicOr(&t.nbm[v >> 5], 1u << (v & 31));
                ++dn;
            }
        } else if (nl[u] < (L)t.Tl) {
            // ids at or above n_big cannot be hubs: no look at the row
            if (v < a.n_big) {
                const uint32_t r0 = a.row_ptr[v];                 // independent of the exchange
                deg[u] = (t.lend ? t.lend[v] : a.row_ptr[v + 1]) - r0;
            }
            // without stamps only hubs join the chunk queue once
            to_near[u] = (t.nostamp && deg[u] < HEAVY_DEG) ||
                         atomicExch(&a.stamp_near[v], t.tag_next) != t.tag_next;
        } else {
            cand[u] = true;      // bounds far_min
            // with the far scan, the split finds far vertices by their labels
            if (!SCAN) to_far[u] = atomicExch(&a.stamp_far[v], t.tag_far) != t.tag_far;
        }
    }
    push_far<SCAN, N>(a, st, t, to_far, cand, vs, [&](int u) {
        return (uint32_t)(NARROW ? nl[u] >> a.lshift : (uint64_t)nl[u] >> 32);
    });
    push_near<N>(a, st, t, flush, to_near, vs, deg);
    if (SCAN && t.dense) {
        dn = __reduce_add_sync(FULL, dn);
        if (lane_id() == 0 && dn) st.dn_near[threadIdx.x >> 5] += dn;
    }
}

// Lists vertex u (lanes with `want`; hdeg arcs in its heavy part) in the
// current band once: as one item, or as CHUNK-arc pieces when the heavy
// part is long.  A vertex without heavy arcs needs no listing.
__device__ __forceinline__ void band_track(const SsspArgs &a, Stage &st, bool want, uint32_t u,
                                           uint32_t hdeg, uint32_t tag) {
    uint32_t listed = 0;     // heavy arcs this lane lists
    if (a.dense) {
        // dense band list: a bit per listed vertex (the pass reads the
        // bitmap), so only the hubs need the stamp that lists them once
        const bool small = want && hdeg > 0 && hdeg < HEAVY_DEG;
        if (small) atomicOr(&a.bbm[u >> 5], 1u << (u & 31));
        const uint32_t c = (uint32_t)__popc(__ballot_sync(FULL, small));
        if (lane_id() == 0 && c) st.dn_band[threadIdx.x >> 5] += c;
        if (small) listed = hdeg;
        want = want && hdeg >= HEAVY_DEG;
    }
    bool add = want && hdeg > 0 && atomicExch(&a.stamp_band[u], tag) != tag;
    const bool big = add && hdeg >= HEAVY_DEG;
    const uint32_t w = threadIdx.x >> 5;
    if (add) listed = hdeg;
    listed = __reduce_add_sync(FULL, listed);
    if (lane_id() == 0 && listed) st.hs[w] += listed;
    region_append(add && !big, u, st.band_buf + w * BAND_REGION, &st.band_n[w], BAND_REGION, true,
                  a.band_q, &a.ctl->band_count, a.n, &a.ctl->err);
    for (uint32_t m = __ballot_sync(FULL, big); m; m &= m - 1) {     // chunk lists: the whole warp
        const uint32_t l = __ffs(m) - 1;
        const uint32_t ul = __shfl_sync(FULL, u, l);
        const uint32_t nc = (__shfl_sync(FULL, hdeg, l) + CHUNK - 1) / CHUNK;
        uint32_t base = 0;
        if (lane_id() == 0) base = atomicAdd(&a.ctl->band_hcount, nc);
        base = __shfl_sync(FULL, base, 0);
        if (base + nc > a.heavy_cap || base + nc < base) {
            if (lane_id() == 0) atomicOr(&a.ctl->err, ERR_CAPACITY);
            continue;
        }
        for (uint32_t c = lane_id(); c < nc; c += 32) a.band_hq[base + c] = ((uint64_t)ul << 32) | c;
    }
}

// Relaxes the arcs of up to 32 rows, one per lane ([s, s + deg), tail label
// lab; lanes without work deg = 0), flattened over the lanes.  The lanes'
// rows are first compacted (no empty row in between), so that the row of
// position j is the number of row starts at or before it: one mask per 32
// positions, not a search by shuffles.  The next group's arc records are
// loaded before this group is relaxed.
template <bool NARROW, bool SCAN>
__device__ __forceinline__ void relax_rows(const SsspArgs &a, Stage &st, const PushTargets &t,
                                           uint32_t s, uint32_t deg,
                                           typename LabelOf<NARROW>::T lab, bool flush,
                                           bool precheck, bool stream, uint32_t wlo, uint32_t whi,
                                           uint32_t &attempts, uint32_t &improved,
                                           bool &narrow_miss) {
    const uint32_t lane = lane_id();
    const uint32_t mask = __ballot_sync(FULL, deg != 0);
    if (mask == 0) return;
    const uint32_t rows = (uint32_t)__popc(mask);
    if (mask != FULL) {
        const uint32_t from = nth_set_bit(mask, lane < rows ? lane : 0);
        s = __shfl_sync(FULL, s, from);
        lab = __shfl_sync(FULL, lab, from);
        deg = __shfl_sync(FULL, deg, from);
        if (lane >= rows) deg = 0;
    }
    const uint32_t incl = warp_inclusive_scan(deg);
    const uint32_t total = __shfl_sync(FULL, incl, 31);
    const uint32_t excl = lane < rows ? incl - deg : INF32;
    const uint32_t base = s - excl;      // arc of position j in row r: base(r) + j
    auto load = [&](uint32_t b, auto &g) {
        constexpr int N = sizeof(g.e) / sizeof(g.e[0]);
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const uint32_t b0 = b + 32 * q, j = b0 + lane;
            // rows that start in this window, and those before it
            const uint32_t before = N == 1 ? 0u : (uint32_t)__popc(__ballot_sync(FULL, excl < b0));
            const uint32_t at = excl - b0;
            const uint32_t starts = __reduce_or_sync(FULL, at < 32 ? 1u << at : 0u);
            const uint32_t row = before + (uint32_t)__popc(starts & (FULL >> (31 - lane))) - 1;
            const uint32_t arc = __shfl_sync(FULL, base, row) + j;
            g.lab[q] = __shfl_sync(FULL, lab, row);
            g.valid[q] = j < total;
            g.e[q] = make_uint2(0, 0);
            // hub chunks are streamed (evict first); short rows may be
            // re-read by later hops and stay cacheable
            if (g.valid[q]) g.e[q] = stream ? __ldcs(&a.adj[arc]) : __ldg(&a.adj[arc]);
        }
    };
    if (total <= 32) {
        // a thin frontier's batch: one arc per lane, a quarter of the
        // instructions (a hop is bound by them as much as by its round trips)
        ArcGroup<NARROW, 1> g;
        load(0, g);
        relax_group<NARROW, SCAN, 1>(a, st, t, g, flush, precheck, wlo, whi, attempts, improved,
                                     narrow_miss);
        return;
    }
    ArcGroup<NARROW, ILP> g;
    load(0, g);
    for (uint32_t b = 0; b < total; b += 32 * ILP) {
        ArcGroup<NARROW, ILP> next;
        const bool more = b + 32 * ILP < total;
        if (more) load(b + 32 * ILP, next);
        relax_group<NARROW, SCAN, ILP>(a, st, t, g, flush, precheck, wlo, whi, attempts, improved,
                                       narrow_miss);
        if (more) g = next;
    }
}

// Shared-memory scratch of a pull pass, one per warp, for the 32 * PULL_ILP
// vertices of a step.
template <bool NARROW>
struct PullScratch {
    typename LabelOf<NARROW>::T best[32 * PULL_ILP];   // best label so far
    uint2 row[32 * PULL_ILP];       // compacted rows: arc base, vertex of the step
    uint8_t near[32 * PULL_ILP];    // the vertex has an unsettled neighbour
};

// Pull form of a band's heavy-arc pass (threshold T, every label below T
// final).  Warps sweep the vertex ids (coalesced labels), or the candidate
// list, 32 * PULL_ILP at a step; a vertex at or above T (unreached included)
// reads the arcs of its heavy part and the labels at their other ends.  The
// step's rows are flattened over the lanes as in relax_rows, the next group's
// arc records loaded before this group's labels are waited for.  The best
// proposal (d(u) + w, rank(u)) from a settled neighbour u is gathered per
// vertex in shared memory and, if it beats the vertex's label, sent as one
// fire-and-forget atomicMin; it bounds far_min as a far push proposal does.
// The sweep also clears the band bitmap that the push form would have read.
// The warps' sums of the heavy arcs met go to st.hs (the pass's cost).
// `out` (sweep of every id, no tail): the unsettled vertices with arcs are
// listed there, the candidates of the split that follows.
// `tail`: the pass starts the unbounded tail band.  A vertex whose neighbours
// are all settled can improve nothing, so the pass reads whole rows, notes
// which vertices have an unsettled neighbour, and pushes those of them that
// are reached (R-MAT 26, degree 8, k = 10,000: 18.5 -> 3.6 M vertices, the
// first tail iteration 0.89 -> 0.48 ms, the pass 2.49 -> 1.31 ms with the
// flattened steps).
template <bool NARROW>
__device__ __noinline__ void pull_pass(const SsspArgs &a, Stage &st, PullScratch<NARROW> *scratch,
                                       uint64_t T, const uint32_t *list, uint32_t count,
                                       uint32_t *out, uint32_t *out_count, bool tail,
                                       uint32_t *nbm, uint32_t *qn, uint32_t *qn_count,
                                       uint64_t *hqn, uint32_t *hqn_count, uint32_t &attempts,
                                       uint32_t &improved, bool &narrow_miss) {
    using L = typename LabelOf<NARROW>::T;
    constexpr L UNREACHED = (L)~0ull;
    const uint32_t lane = lane_id();
    const uint32_t wib = threadIdx.x >> 5;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    PullScratch<NARROW> &sc = scratch[wib];
    const L Tl = (L)threshold_label<NARROW>(a, T);
    // where the tail's first frontier goes (light vertices as bits when dense)
    PushTargets t;
    t.qn = qn;
    t.qn_count = qn_count;
    t.hqn = hqn;
    t.hqn_count = hqn_count;
    t.dense = a.dense != 0;
    t.nbm = nbm;
    t.nostamp = false;
    t.nostamp_stamp = nullptr;
    t.tag_next = 0;
    t.hsum = nullptr;
    t.lend = nullptr;
    uint32_t met = 0;
    L fmin = UNREACHED;
    // the vertices: every id that may have arcs, or the candidate list (then
    // the band bitmap is cleared by a sweep of its own)
    if (list && a.dense)
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n_words;
             i += gridDim.x * blockDim.x)
            if (ldcg_u32(&a.bbm[i])) a.bbm[i] = 0;
    const uint32_t nv = list ? count : a.n_live;
    for (uint32_t b = warp * 32 * PULL_ILP; b < nv; b += nwarps * 32 * PULL_ILP) {
        if (!list && a.dense && lane < PULL_ILP && (b >> 5) + lane < a.n_words &&
            ldcg_u32(&a.bbm[(b >> 5) + lane]))
            a.bbm[(b >> 5) + lane] = 0;
        uint32_t vs[PULL_ILP];
        L lab[PULL_ILP];
        uint32_t s[PULL_ILP], r1[PULL_ILP], r0[PULL_ILP];
#pragma unroll
        for (int c = 0; c < PULL_ILP; ++c) {
            const uint32_t i = b + 32u * c + lane;
            vs[c] = i < nv ? (list ? ldcg_u32(&list[i]) : i) : INF32;
        }
#pragma unroll
        for (int c = 0; c < PULL_ILP; ++c)    // past the end: taken as settled
            lab[c] = vs[c] != INF32 ? raw_label<NARROW>(a, vs[c]) : (L)0;
        bool uns[PULL_ILP];
#pragma unroll
        for (int c = 0; c < PULL_ILP; ++c) {
            const uint32_t v = vs[c];
            s[c] = r1[c] = r0[c] = 0;
            uns[c] = lab[c] >= Tl;
            if (uns[c]) {
                r1[c] = a.row_ptr[v + 1];
                r0[c] = a.row_ptr[v];
                s[c] = a.lend ? a.lend[v] : r0[c];
            }
            sc.best[32 * c + lane] = lab[c];
            sc.near[32 * c + lane] = 0;
        }
        if (out) {
            // the sweep over every id lists the unsettled vertices with arcs
            // (the candidates of the split that follows), staged in the band
            // regions, which a heavy-arc pass does not use
#pragma unroll
            for (int c = 0; c < PULL_ILP; ++c)
                region_append(uns[c] && r1[c] != r0[c], vs[c], st.band_buf + wib * BAND_REGION,
                              &st.band_n[wib], BAND_REGION, true, out, out_count, a.n,
                              &a.ctl->err);
        }
        // the step's rows, compacted: rows with arcs in order, their first
        // positions in excl
        uint32_t excl[PULL_ILP], rows = 0, total = 0;
#pragma unroll
        for (int c = 0; c < PULL_ILP; ++c) {
            met += r1[c] - s[c];
            const uint32_t from = tail ? r0[c] : s[c], deg = r1[c] - from;
            const uint32_t m = __ballot_sync(FULL, deg != 0);
            const uint32_t incl = warp_inclusive_scan(deg);
            excl[c] = deg ? total + incl - deg : INF32;
            if (deg)
                sc.row[rows + (uint32_t)__popc(m & lanemask_lt())] =
                    make_uint2(from - excl[c], 32u * c + lane);
            rows += (uint32_t)__popc(m);
            total += __shfl_sync(FULL, incl, 31);
        }
        __syncwarp();
        uint32_t before = 0;           // rows that start before the window
        auto load = [&](uint32_t j0, uint2 (&e)[ILP], uint32_t (&slot)[ILP]) {
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                const uint32_t w0 = j0 + 32 * q, j = w0 + lane;
                uint32_t starts = 0;
#pragma unroll
                for (int c = 0; c < PULL_ILP; ++c)
                    if (excl[c] - w0 < 32) starts |= 1u << (excl[c] - w0);
                starts = __reduce_or_sync(FULL, starts);
                const uint32_t row = before + (uint32_t)__popc(starts & (FULL >> (31 - lane))) - 1;
                before += (uint32_t)__popc(starts);
                e[q] = make_uint2(0, 0);                  // weight 0: no arc
                slot[q] = 0;
                if (j < total) {
                    const uint2 r = sc.row[row];
                    slot[q] = r.y;
                    e[q] = __ldcs(&a.adj[r.x + j]);       // read once per pass: streamed
                }
            }
        };
        uint2 e[ILP];
        uint32_t slot[ILP];
        if (total) load(0, e, slot);
        for (uint32_t j0 = 0; j0 < total; j0 += 32 * ILP) {
            L tl[ILP];
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                tl[q] = 0;
                if (e[q].y && (tail || e[q].y >= a.delta)) tl[q] = raw_label<NARROW>(a, e[q].x);
            }
            uint2 en[ILP];
            uint32_t sn[ILP];
            const bool more = j0 + 32 * ILP < total;
            if (more) load(j0 + 32 * ILP, en, sn);
#pragma unroll
            for (int q = 0; q < ILP; ++q) {
                // an unsettled (or unreached) neighbour proposes nothing yet
                if (tl[q] >= Tl) {
                    sc.near[slot[q]] = 1;
                } else if (e[q].y && e[q].y >= a.delta) {
                    ++attempts;
                    L nl;
                    if constexpr (NARROW) {
                        const uint64_t sum = (uint64_t)e[q].y * a.lstep + tl[q];
                        nl = (uint32_t)sum;
                        if (sum >= a.lmiss) {
                            // only an unreached vertex could take it (a narrow
                            // label holds no such distance): the host
                            // reruns the query with 64-bit labels
                            if (sc.best[slot[q]] == UNREACHED) narrow_miss = true;
                            continue;
                        }
                    } else {
                        const uint64_t nd = (tl[q] >> 32) + (uint64_t)e[q].y;
                        if (nd >= INF32) continue;        // the scan reports the overflow
                        nl = (nd << 32) | (tl[q] & 0xFFFFFFFFull);
                    }
                    if constexpr (NARROW) {
                        if (nl < *(volatile uint32_t *)&sc.best[slot[q]]) atomicMin(&sc.best[slot[q]], nl);
                    } else {
                        auto *best = reinterpret_cast<unsigned long long *>(&sc.best[slot[q]]);
                        if (nl < *(volatile unsigned long long *)best) atomicMin(best, (unsigned long long)nl);
                    }
                }
            }
            if (more) {
#pragma unroll
                for (int q = 0; q < ILP; ++q) {
                    e[q] = en[q];
                    slot[q] = sn[q];
                }
            }
        }
        __syncwarp();
        // each lane settles its own vertices: one atomic per improved one
        bool push[PULL_ILP];
        uint32_t pdeg[PULL_ILP];
#pragma unroll
        for (int c = 0; c < PULL_ILP; ++c) {
            push[c] = false;
            pdeg[c] = 0;
            const L best = sc.best[32 * c + lane];
            if (uns[c] && best < lab[c]) {
                if constexpr (NARROW) atomicMin(&a.label32[vs[c]], best);
                else atomicMin(reinterpret_cast<unsigned long long *>(&a.label[vs[c]]),
                               (unsigned long long)best);
                ++improved;
                fmin = min(fmin, best);
            }
            if (tail) {
                // reached, unsettled and next to an unsettled vertex: the
                // tail's first frontier, whole rows
                const bool want = uns[c] && best != UNREACHED && sc.near[32 * c + lane];
                const uint32_t deg = r1[c] - r0[c];
                const bool bit = t.dense && want && deg < HEAVY_DEG;
                const uint32_t word = __ballot_sync(FULL, bit);
                if (!list) {
                    if (lane == 0 && word) t.nbm[(b + 32u * c) >> 5] = word;
                } else if (bit) {
                    atomicOr(&t.nbm[vs[c] >> 5], 1u << (vs[c] & 31));
                }
                if (lane == 0 && word) st.dn_near[wib] += (uint32_t)__popc(word);
                push[c] = want && !bit;
                pdeg[c] = deg;
            }
        }
        if (tail) push_near<PULL_ILP>(a, st, t, true, push, vs, pdeg);
        __syncwarp();
    }
    met = __reduce_add_sync(FULL, met);
    uint32_t fd = fmin == UNREACHED ? INF32 : (uint32_t)(NARROW ? fmin >> a.lshift : (uint64_t)fmin >> 32);
    fd = __reduce_min_sync(FULL, fd);
    if (lane == 0) {
        st.hs[wib] += met;
        if (fd != INF32) atomicMin(&st.far_min, fd);
    }
}

// ---------------------------------------------------------------------------
// the persistent near/far kernel
// ---------------------------------------------------------------------------

// SCAN: splits scan the labels (a.far_scan), else there is a far pile.
// BLOCKS per SM: three (80 registers, 318 to 378 bytes of spill stores), or two:
// the far-pile forms then spill nothing, the label-scan forms 122 (narrow) and
// 216 bytes.
constexpr int SSSP_BLOCKS = 3;
template <bool NARROW, bool SCAN, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS) sssp_kernel(const __grid_constant__ SsspArgs a) {
    __shared__ Stage st;
    __shared__ PushTargets t;      // this iteration's (shared: off the hot loops' registers)
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    Control *ctl = a.ctl;
    uint32_t attempts = 0, improved = 0;      // this thread's
    bool narrow_miss = false;
    // trace: each warp's counter sums at the start of the iteration (lane 0
    // keeps them in shared memory, off the registers of the hot loops)
    __shared__ unsigned long long trace_snap[SSSP_WARPS][3];
    if (threadIdx.x < SSSP_WARPS * 3) (&trace_snap[0][0])[threadIdx.x] = 0;
    uint32_t it = 0, phase = 0, bands = 0;
    // T: the threshold; Tb: the end of the band (T is below it in the first
    // band's first step)
    uint64_t Tb = a.delta, T = a.step0 && a.step0 < a.delta ? a.step0 : a.delta, T_old = 0;
    bool first = (blockIdx.x == 0 && threadIdx.x == 0);
    bool hp = false;               // this iteration is a band's heavy-arc pass
    bool pull = false;             // ... in the pull form
    // With the far scan, the first split lists every vertex left unsettled
    // (those with arcs); later splits and pull passes visit that list,
    // which each split shrinks, instead of every id.
    bool listed = false;
    // Tail: after a band whose heavy-arc pass ran in the pull form (it
    // settled most of the graph's heavy arcs), the rest runs as one
    // unbounded band, a frontier Bellman-Ford over whole rows: on a
    // small-world graph the unsettled vertices hang off the settled core
    // by short chains, and a few iterations reach the fixed point that a
    // band per delta would approach in many splits.
    bool tail = false;
    __shared__ PullScratch<NARROW> pull_scratch[SCAN ? SSSP_WARPS : 1];
    // heavy arcs a pull pass would read now, bounded from above: all arcs
    // at first, then what the last pull pass met (the unsettled set only
    // shrinks)
    __shared__ unsigned long long pull_bound;
    if (threadIdx.x == 0) pull_bound = a.m;
    bool cur_dense = false;        // this iteration's light items are the bits of a near bitmap

    // This iteration's frontier, read when its last push was known to be in;
    // split: it also splits the far pile, whose sizes are n_far and f_min.
    uint32_t n_light = min(ldcg_u32(&ctl->near_count[0]), a.n);
    uint32_t n_heavy = min(ldcg_u32(&ctl->heavy_count[0]), a.heavy_cap);
    uint32_t n_far = 0;
    bool split = false;
    uint32_t bar_target = 0;

    for (;;) {
        const uint32_t cs = it % 3, ns = (it + 1) % 3;
        if (first) {
            ctl->near_count[(it + 2) % 3] = 0;
            ctl->heavy_count[(it + 2) % 3] = 0;
            ctl->work_next[(it + 2) % 3] = 0;
            if (hp && pull) ++ctl->pulls;
            ctl->trace_warps = nwarps;
            if (it < TRACE_LEN) {
                ctl->trace[it][0] = n_light;
                ctl->trace[it][1] = n_heavy;
                ctl->trace[it][2] = split ? n_far : ldcg_u32(&ctl->far_count[phase % 3]);
                ctl->trace[it][3] = (uint32_t)T;
                ctl->trace_ns[it] = global_ns();
            }
        }
        const bool odd = it & 1;
        const uint32_t *qc = hp ? a.band_q : (odd ? a.q1 : a.q0);
        const uint64_t *hqc = hp ? a.band_hq : (odd ? a.hq1 : a.hq0);
        // fc: which of the two piles takes this phase's far vertices; fs: its
        // counters (three, so that one can be cleared while the piles of two
        // phases are in use)
        const uint32_t fc = phase & 1, fs = phase % 3;
        // dense in: light items from this iteration's near bitmap (or, in a
        // dense heavy-arc pass, the band bitmap); dense out: a large
        // frontier (a fraction of the graph, or many hub chunks) pushes its
        // light vertices as bits for the next iteration.  Every block reads
        // the same counts, so all agree.
        const bool dense_in = hp ? a.dense != 0 : cur_dense;
        const bool push_dense =
            a.dense && !hp && (n_light >= a.n / 128 || n_heavy >= a.n / 4096);
        uint32_t *bm_in = hp ? a.bbm : ((it & 1) ? a.nbm1 : a.nbm0);
        // arcs relaxed by this iteration: all; light ones while a band
        // iterates under the split; heavy ones in the band's closing pass
        // (in the tail every relaxation covers whole rows)
        const uint32_t wlo = hp ? a.delta : 0u;
        const uint32_t whi = (a.defer && !hp && !tail) ? a.delta : 0xFFFFFFFFu;
        const bool track = a.defer && !hp && !tail;
        const uint32_t *lend = tail ? nullptr : a.lend;
        // warp-local rounds; a frontier thinner than the grid takes some in
        // any case (with the far pile and whole rows)
        const uint32_t local_rounds =
            hp ? 0u : a.local_rounds ? a.local_rounds
                    : !SCAN && !a.defer && n_light + n_heavy < a.thin ? a.thin_rounds : 0u;
        const uint32_t tag_band = a.base_band + bands;
        if (threadIdx.x == 0) {
            t.qn = odd ? a.q0 : a.q1;
            t.qn_count = &ctl->near_count[ns];
            t.hqn = odd ? a.hq0 : a.hq1;
            t.hqn_count = &ctl->heavy_count[ns];
            t.farq = fc ? a.far1 : a.far0;
            t.far_count = &ctl->far_count[fs];
            t.far_min = &ctl->far_min[fs];
            // a pull pass without a list yet sweeps every id and lists the
            // unsettled ones as this phase's pile (empty with the far scan)
            t.bandq = hp && pull ? t.farq : a.band_q;
            t.band_count = hp && pull ? t.far_count : &ctl->band_count;
            t.tag_next = a.base_near + it + 1;
            t.tag_far = a.base_far + phase;
            t.Tl = threshold_label<NARROW>(a, T);
            t.dense = push_dense;
            t.nbm = odd ? a.nbm0 : a.nbm1;
            t.nostamp = local_rounds != 0;
            t.nostamp_stamp = a.stamp_near;
            t.lend = lend;
            t.hsum = track ? &ctl->band_hsum : (hp && pull ? &ctl->pull_hsum : nullptr);
        }
        stage_reset(st);
        // Vertices per warp batch: a thin frontier is spread over all warps
        // (fewer sequential rounds per warp), a thick one packs 32 per warp.
        uint32_t per = (n_light + nwarps - 1) / nwarps;
        uint32_t bsz = per <= 1 ? 1 : per <= 2 ? 2 : per <= 4 ? 4 : per <= 8 ? 8 : per <= 16 ? 16 : 32;
        // A dense work item is a vertex range of about equal arcs (a range
        // of equal vertices gave the first warps 256 rows of nearly
        // HEAVY_DEG arcs each: on R-MAT 16, k = 16 the slowest warp of an
        // iteration was busy 1.2 ms against a mean of 11 us, and the query
        // took 3.6 ms against 0.87).  A sparse
        // bitmap (under one set bit per two words) is read in the coarser
        // ranges: the sweep itself is then the cost.
        const bool sparse = n_light < a.n_words / 2;
        const uint32_t *items = sparse ? a.sparse_items : a.items;
        // Few hub chunks are cut in SUB_CHUNKS pieces of one relax_group each.
        const uint32_t subs = n_heavy * SUB_CHUNKS <= nwarps ? SUB_CHUNKS : 1u;
        const uint32_t n_hitems = n_heavy * subs;
        const uint32_t n_work = n_hitems + (dense_in ? (sparse ? a.n_sparse_items : a.n_items)
                                                     : (n_light + bsz - 1) / bsz);
        if (a.trace && lane == 0) trace_snap[threadIdx.x >> 5][2] = global_ns();
        if (!SCAN && split) {
            // The pile of the phase that this iteration ended (see the
            // decision below): a vertex below the old threshold was settled
            // while parked; one below the new threshold joins the next
            // frontier, the rest the new pile.  Vertices that this
            // iteration's relaxations push as well are kept apart by the
            // stamps (a region without stamps may hold a vertex twice).
            // Before the frontier, and the pile dealt out to the warps one
            // vertex each in turn, so that the warp-local rounds follow its
            // vertices at once, on all warps alike (grid 4096 x 4096, 32
            // rounds: 9.2 ms split after the rounds, 8.1 before them, 7.8
            // with the early split; from pieces of 32 the few warps that had
            // one held up the others, 12.1).
            const uint32_t *pile = fc ? a.far0 : a.far1;
            for (uint64_t b = 0; b * nwarps + warp < n_far; b += 32 * SPLIT_ILP) {
                uint32_t v[SPLIT_ILP], deg[SPLIT_ILP];
                uint64_t d[SPLIT_ILP];
                bool to_near[SPLIT_ILP], keep[SPLIT_ILP], to_far[SPLIT_ILP];
#pragma unroll
                for (int c = 0; c < SPLIT_ILP; ++c) {
                    const uint64_t i = (b + 32u * c + lane) * nwarps + warp;
                    v[c] = i < n_far ? ldcg_u32(&pile[i]) : INF32;
                }
#pragma unroll
                for (int c = 0; c < SPLIT_ILP; ++c)
                    d[c] = v[c] != INF32 ? sssp_label<NARROW>(a, v[c]) >> 32 : 0ull;
#pragma unroll
                for (int c = 0; c < SPLIT_ILP; ++c) {
                    to_near[c] = d[c] >= T_old && d[c] < T;
                    deg[c] = 0;
                    if (to_near[c]) {
                        if (v[c] < a.n_big) deg[c] = a.row_ptr[v[c] + 1] - a.row_ptr[v[c]];
                        if (!t.nostamp || deg[c] >= HEAVY_DEG)
                            to_near[c] = atomicExch(&a.stamp_near[v[c]], t.tag_next) != t.tag_next;
                    }
                    keep[c] = d[c] >= T;
                    to_far[c] = keep[c] && atomicExch(&a.stamp_far[v[c]], t.tag_far) != t.tag_far;
                }
                push_far<SCAN, SPLIT_ILP>(a, st, t, to_far, keep, v, [&](int c) { return (uint32_t)d[c]; });
                push_near<SPLIT_ILP>(a, st, t, !t.nostamp, to_near, v, deg);
            }
        }
        if (SCAN && hp && pull) {
            uint32_t *pile = fc ? a.far1 : a.far0;
            // with the tail to follow, the pass pushes its first frontier
            pull_pass<NARROW>(a, st, pull_scratch, T, listed ? pile : nullptr,
                              listed ? min(ldcg_u32(&ctl->far_count[fs]), a.n) : a.n,
                              (listed || a.tail) ? nullptr : pile, &ctl->far_count[fs],
                              a.tail != 0, t.nbm, t.qn, t.qn_count, t.hqn, t.hqn_count,
                              attempts, improved, narrow_miss);
        } else {
            // The last quarter of a long list is handed out on demand (the
            // next index is fetched while an item is relaxed), so that the
            // iteration does not end with its slowest warp (R-MAT 26, degree
            // 8, k = 10,000: the thickest iterations 3.2 ms, all fixed 3.65).
            // After the list come the warp-local rounds (the vertices this
            // warp staged for the next iteration, relaxed right away, a hop
            // further per round, without a barrier; what is left is
            // flushed).  One loop for all of them: the relaxation is
            // expanded once.
            const uint32_t n_fixed = n_work < 8 * nwarps ? n_work : n_work / 4 * 3 / nwarps * nwarps;
            const uint32_t wib = threadIdx.x >> 5;
            const uint32_t *region = st.near_buf + wib * NEAR_REGION;
            uint32_t rounds = local_rounds;
            uint32_t wi = warp, grab = 0, local_lo = 0;
            for (;;) {
                // this item: nb batches of up to 32 vertices
                const bool hub = wi < n_hitems, local = wi >= n_work;
                uint32_t nb = 1, word = 0, excl = 0, total = 0, w0 = 0, local_hi = 0;
                if (local) {
                    if (rounds == 0) break;
                    --rounds;
                    __syncwarp();
                    local_hi = min(*(volatile uint32_t *)&st.near_n[wib], NEAR_REGION);
                    // (a thin frontier that grew past a batch goes back to
                    // the queue: the other warps take their share)
                    if (local_lo >= local_hi || (local_hi - local_lo > 32 && !a.local_rounds)) break;
                    nb = (local_hi - local_lo + 31) / 32;
                } else {
                    if (wi + nwarps >= n_fixed && n_fixed != n_work && lane == 0)
                        grab = atomicAdd(&ctl->work_next[cs], 1u);
                    if (SCAN && dense_in && !hub) {
                        // the words of the item's vertex range, one per lane
                        // (the range's bits are read and cleared; a word may
                        // be shared with the neighbouring items); their set
                        // bits, 32 at a time, are the vertices
                        const uint32_t v0 = __ldg(&items[wi - n_hitems]);
                        const uint32_t v1 = __ldg(&items[wi - n_hitems + 1]);
                        const uint32_t w1 = (v1 - 1) >> 5;
                        w0 = v0 >> 5;
                        if (w0 + lane <= w1) {
                            uint32_t own = FULL;
                            if (lane == 0) own <<= v0 & 31;
                            if (w0 + lane == w1) own &= FULL >> (31 - ((v1 - 1) & 31));
                            word = ldcg_u32(&bm_in[w0 + lane]) & own;
                            if (word) {
                                if (own == FULL) bm_in[w0 + lane] = 0;
                                else atomicAnd(&bm_in[w0 + lane], ~own);
                            }
                        }
                        const uint32_t cnt = (uint32_t)__popc(word);
                        excl = warp_inclusive_scan(cnt);
                        total = __shfl_sync(FULL, excl, 31);
                        excl -= cnt;
                        nb = (total + 31) / 32;
                    }
                }
                for (uint32_t b = 0; b < nb; ++b) {
                    // one vertex per lane; a hub chunk (or a piece of one) is
                    // part of one row, on lane 0
                    bool has;
                    uint32_t u = 0, c = 0, sub = 0;
                    if (local) {
                        const uint32_t i = local_lo + 32 * b + lane;
                        has = i < local_hi;
                        if (has) u = region[i];
                    } else if (hub) {
                        has = lane == 0;
                        if (has) {
                            const uint64_t item = __ldcg(reinterpret_cast<const unsigned long long *>(
                                &hqc[subs > 1 ? wi / SUB_CHUNKS : wi]));
                            sub = subs > 1 ? wi % SUB_CHUNKS : 0u;
                            u = (uint32_t)(item >> 32);
                            c = (uint32_t)item;
                        }
                    } else if (SCAN && dense_in) {
                        const uint32_t j = 32 * b + lane;
                        has = j < total;
                        const uint32_t owner = warp_owner_search(excl, has ? j : 0);
                        const uint32_t wo = __shfl_sync(FULL, word, owner);
                        const uint32_t eo = __shfl_sync(FULL, excl, owner);
                        if (has) u = (w0 + owner) * 32 + nth_set_bit(wo, j - eo);
                    } else {
                        // bsz frontier vertices per warp
                        const uint32_t i = (wi - n_hitems) * bsz + lane;
                        has = lane < bsz && i < n_light;
                        if (has) u = ldcg_u32(&qc[i]);
                    }
                    uint32_t s = 0, deg = 0, hdeg = 0;
                    auto lab = (typename LabelOf<NARROW>::T)~0ull;
                    if (has) {
                        const uint32_t r0 = a.row_ptr[u], r1 = a.row_ptr[u + 1];
                        const uint32_t le = lend ? lend[u] : r1;      // light part [r0, le)
                        // (a warp-local round needs no more than the current
                        // label: every later improvement of u appends u
                        // again, to the improving warp's region)
                        lab = raw_label<NARROW>(a, u);
                        // the closing pass of a band covers the heavy part
                        // (or the whole row), else the light one
                        s = hp && lend ? le : r0;
                        deg = (hp ? r1 : le) - s;
                        if (!hp) hdeg = lend ? r1 - le : r1 - r0;
                        if (hub) {
                            const uint32_t at = c * CHUNK + sub * (CHUNK / SUB_CHUNKS);
                            s += at;
                            deg = deg > at ? min(deg - at, CHUNK / subs) : 0u;
                        }
                        if (lab == (typename LabelOf<NARROW>::T)~0ull) deg = 0;
                    }
                    if (track) band_track(a, st, has && (c | sub) == 0, u, hdeg, tag_band);
                    relax_rows<NARROW, SCAN>(a, st, t, s, deg, lab, !local,
                                             hub || (SCAN && dense_in) || (!local && bsz == 32), hub,
                                             wlo, whi, attempts, improved, narrow_miss);
                }
                if (local) local_lo = local_hi;
                else wi = wi + nwarps < n_fixed || n_fixed == n_work ? wi + nwarps
                                                                     : n_fixed + __shfl_sync(FULL, grab, 0);
            }
            if (lane == 0) st.local_lo[wib] = local_lo;
        }
        if (a.trace && it < TRACE_LEN) {
            // per warp: busy time of this iteration's relaxation (sum, max)
            unsigned long long da = attempts, di = improved;
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                da += __shfl_xor_sync(FULL, da, o);
                di += __shfl_xor_sync(FULL, di, o);
            }
            if (lane == 0) {
                unsigned long long *snap = trace_snap[threadIdx.x >> 5];
                const unsigned long long busy = global_ns() - snap[2];
                const unsigned long long sa = da, si = di;
                da -= snap[0];
                di -= snap[1];
                snap[0] = sa;
                snap[1] = si;
                if (da | di) {
                    atomicAdd(&ctl->trace_relax[it][0], da);
                    atomicAdd(&ctl->trace_relax[it][1], di);
                }
                atomicAdd(&ctl->trace_busy[it][0], busy);
                atomicMax(&ctl->trace_busy[it][1], busy);
            }
        }
        flush_stage(st, t, a.n, &ctl->err);
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) {
            if (first) ctl->exit_reason = 3;
            break;
        }
        // a pull pass that starts the tail set its frontier's bits (dense)
        cur_dense = (hp && pull && a.tail) ? a.dense != 0 : push_dense;
        ++it;
        const bool was_hp = hp;
        if (hp) {
            ++bands;               // later listings use a fresh tag
            hp = false;
            if (pull && a.tail) {
                // the tail band: no threshold, whole rows, no more splits
                tail = true;
                T = INF32;
                if (first) ctl->tail_it = it;
            }
            if (pull) {
                // every thread has read pull_bound at the decision, a
                // barrier ago; one writes the new bound, read at the next
                if (threadIdx.x == 0)
                    pull_bound = ldcg_u64(reinterpret_cast<const uint64_t *>(&ctl->pull_hsum));
                listed = true;     // the pass listed the candidates (or used the list)
            }
            pull = false;
        }
        if (it >= a.max_iters) {
            if (first) {
                atomicOr(&ctl->err, ERR_TIMEOUT);
                ctl->exit_reason = 2;
            }
            break;
        }
        n_light = min(ldcg_u32(&ctl->near_count[ns]), a.n);
        n_heavy = min(ldcg_u32(&ctl->heavy_count[ns]), a.heavy_cap);
        const uint32_t far_now = ldcg_u32(&ctl->far_count[fs]);   // stable if the pile is split next
        const uint32_t fmin_now = ldcg_u32(&ctl->far_min[fs]);
        split = false;
        if (!SCAN && !a.defer) {
            // Far pile, no light/heavy split: the next iteration splits the
            // pile as well (no iteration and barrier of its own) when the
            // frontier drained, and already when it is thin (a.thin): the
            // grid's warps would idle through the last hops of every band.
            // Every block decides on near_count, which no iteration writes
            // before all have read it.  A thin frontier
            // always ends the phase (the threshold stays if the pile is
            // empty): an ended phase's pile takes no more pushes, so every
            // block reads the same count and minimum of it.
            if (n_light + n_heavy >= a.thin) continue;
            const bool drained = (n_light | n_heavy) == 0;
            n_far = min(far_now, a.n);
            if (drained && n_far == 0) {
                if (first) ctl->exit_reason = 1;       // converged
                break;
            }
            ++phase;
            if (first) {           // last read a phase ago, next used a phase from now
                ctl->far_count[(phase + 1) % 3] = 0;
                ctl->far_min[(phase + 1) % 3] = INF32;
            }
            if (n_far) {
                if (first) atomicAdd(&ctl->advances, 1u);
                T_old = T;
                T = (fmin_now != INF32 && (uint64_t)fmin_now > T ? (uint64_t)fmin_now : T) +
                    a.delta;
                split = true;
            }
            continue;
        }
        if (n_light | n_heavy) continue;
        if (tail) {                    // the tail's frontier drained: converged
            if (first) ctl->exit_reason = 1;
            break;
        }
        // The first band is reached in two steps (a.step0, then its end): a
        // vertex reached by long light paths is then relaxed when the nearer
        // ones have settled, not once per improvement.  The band's listings
        // go on; its heavy arcs follow at its end.
        const bool step = SCAN && !was_hp && T < Tb && fmin_now < Tb;
        if (SCAN && T < Tb && !step) T = Tb;           // nothing is left below the band's end
        // Band drained: its heavy arcs first (one more iteration), then the
        // split.  The band lists are cleared in the split, so no block can
        // still be reading their counts here.
        // The pull form when the band listed more heavy arcs than a pull
        // would read: the heavy arcs of the vertices unsettled before the
        // band less the band's own, plus the sweep over every label (taken
        // as n / 8 arcs: coalesced, against one random label per arc).
        // Listings count a vertex once per relaxation, which leans to the
        // pull only when the band is large.
        if (a.defer && !was_hp && !tail && !step &&
            (ldcg_u32(&ctl->band_count) | ldcg_u32(&ctl->band_hcount)) != 0) {
            hp = true;
            n_light = min(ldcg_u32(&ctl->band_count), a.n);
            n_heavy = min(ldcg_u32(&ctl->band_hcount), a.heavy_cap);
            const unsigned long long listed_hs =
                ldcg_u64(reinterpret_cast<const uint64_t *>(&ctl->band_hsum));
            const unsigned long long rest = pull_bound > listed_hs ? pull_bound - listed_hs : 0ull;
            const uint32_t sweep =
                listed ? min(far_now, a.n) : a.n;
            pull = a.pull == 2 || (a.pull == 1 && listed_hs > rest + sweep / 8);
            continue;
        }

        // Near frontier drained: raise the threshold and split the far pile.
        // Every block has just read near_count[it % 3] to take this branch,
        // so the split must not push there: it fills the slot (and queue)
        // of iteration it + 1, and the loop resumes at it + 1.  That slot was
        // cleared at the top of iteration it - 1 and nothing reads it before
        // the barrier that ends the split.  Iteration it + 1 will push into
        // slot (it + 2) % 3, which the skipped top of iteration it would
        // have cleared: clear it here (its last reader was iteration it - 1).
        // With the far scan there is no pile: every label at or above the
        // threshold came from a proposal (or a split) that lowered far_min,
        // so an infinite far_min means no vertex is left unsettled.
        const uint32_t nf = min(far_now, a.n), fmin = fmin_now;
        if (SCAN ? fmin == INF32 : nf == 0) {           // converged
            if (first) ctl->exit_reason = 1;
            break;
        }
        T_old = T;
        if (step) {
            T = Tb;
        } else {
            T = Tb = (fmin != INF32 && (uint64_t)fmin > T ? (uint64_t)fmin : T) + a.delta;
        }
        ++phase;
        const uint32_t *pile = fc ? a.far1 : a.far0;
        const uint32_t fsn = phase % 3;        // the new phase's far counters
        const uint32_t its = it + 1;
        if (first) {
            ctl->near_count[(its + 1) % 3] = 0;
            ctl->heavy_count[(its + 1) % 3] = 0;
            ctl->work_next[(its + 1) % 3] = 0;
            atomicAdd(&ctl->advances, 1u);
            if (!step) {
                ctl->band_count = 0;
                ctl->band_hcount = 0;
                ctl->band_hsum = 0;
            }
            ctl->far_count[(phase + 1) % 3] = 0;   // last read a phase ago
            ctl->far_min[(phase + 1) % 3] = INF32;
        }
        // the first split sweeps every id, and sets whole bitmap words;
        // a split over the list sets bits, and only for a list long enough
        // that the next iteration's sweep of the bitmap pays
        const bool from_list = SCAN && listed;
        const bool dense_out = a.dense && (!from_list || nf >= a.n / 64);
        if (threadIdx.x == 0) {
            t.qn = (its & 1) ? a.q1 : a.q0;
            t.qn_count = &ctl->near_count[its % 3];
            t.hqn = (its & 1) ? a.hq1 : a.hq0;
            t.hqn_count = &ctl->heavy_count[its % 3];
            t.farq = fc ? a.far0 : a.far1;
            t.far_count = &ctl->far_count[fsn];
            t.far_min = &ctl->far_min[fsn];
            // With the far scan the split rebuilds the pile as the candidate
            // list: every vertex at or above T_old (the new band's frontier
            // and all later ones; unreached vertices with arcs too), staged
            // in the band regions, which no band listing uses during a
            // split.
            t.bandq = SCAN ? t.farq : a.band_q;
            t.band_count = SCAN ? t.far_count : &ctl->band_count;
            t.tag_next = a.base_near + its;
            t.tag_far = a.base_far + phase;
            t.dense = dense_out;
            t.nbm = (its & 1) ? a.nbm1 : a.nbm0;
            t.nostamp = false;             // the split visits each vertex once
            t.hsum = nullptr;
            t.lend = a.lend;
        }
        stage_reset(st);
        // the far pile (or list), or with the far scan first every vertex
        const uint32_t n_split = (SCAN && !from_list) ? a.n_live : nf;
        // SPLIT_ILP chunks of 32 per warp step, their loads issued together.
        // A vertex is met once here (the pile holds it once, the scan visits
        // each id once) and nothing relaxes during the split, so its near
        // stamp is a plain store.
        for (uint32_t b = warp * 32 * SPLIT_ILP; b < n_split; b += nwarps * 32 * SPLIT_ILP) {
            uint32_t v[SPLIT_ILP], deg[SPLIT_ILP];
            uint64_t d[SPLIT_ILP];
            bool to_near[SPLIT_ILP], cand[SPLIT_ILP], keep[SPLIT_ILP], in[SPLIT_ILP];
#pragma unroll
            for (int c = 0; c < SPLIT_ILP; ++c) {
                const uint32_t i = b + 32u * c + lane;
                in[c] = i < n_split;
                v[c] = 0;
                d[c] = INF32;
                if (in[c]) v[c] = (SCAN && !from_list) ? i : ldcg_u32(&pile[i]);
            }
#pragma unroll
            for (int c = 0; c < SPLIT_ILP; ++c)
                if (in[c]) d[c] = sssp_label<NARROW>(a, v[c]) >> 32;
#pragma unroll
            for (int c = 0; c < SPLIT_ILP; ++c) {
                const bool valid = d[c] != INF32;                  // unreached or past the end
                to_near[c] = valid && d[c] >= T_old && d[c] < T;   // below T_old: already settled
                cand[c] = valid && d[c] >= T;
                deg[c] = 0;
                // dense: ids at or above n_big are light without a look at the row
                if (to_near[c] && (!a.dense || v[c] < a.n_big)) {
                    const uint32_t r0 = a.row_ptr[v[c]];
                    const uint32_t r1 = t.lend ? t.lend[v[c]] : a.row_ptr[v[c] + 1];
                    a.stamp_near[v[c]] = t.tag_next;
                    deg[c] = r1 - r0;
                }
                if (SCAN) {
                    // the list keeps to_near and cand vertices, and unreached
                    // ones with arcs (isolated vertices are never reached)
                    keep[c] = to_near[c] || cand[c];
                    if (step && !from_list) keep[c] = false;       // the band's closing lists them
                    else if (in[c] && !valid)
                        keep[c] = from_list || a.row_ptr[v[c] + 1] != a.row_ptr[v[c]];
                } else {
                    keep[c] = cand[c] &&
                              atomicExch(&a.stamp_far[v[c]], t.tag_far) != t.tag_far;
                }
            }
            bool push[SPLIT_ILP];
#pragma unroll
            for (int c = 0; c < SPLIT_ILP; ++c) {
                // dense: light vertices as bits; from the id sweep a chunk is
                // one bitmap word (empty since the band drained), so one store
                const bool bit = dense_out && to_near[c] && deg[c] < HEAVY_DEG;
                const uint32_t word = __ballot_sync(FULL, bit);
                if (from_list) {
                    if (bit) atomicOr(&t.nbm[v[c] >> 5], 1u << (v[c] & 31));
                } else if (lane == 0 && word) {
                    t.nbm[(b + 32u * c) >> 5] = word;
                }
                if (lane == 0 && word) st.dn_near[threadIdx.x >> 5] += (uint32_t)__popc(word);
                push[c] = to_near[c] && !bit;
                if (SCAN) {
                    const uint32_t w = threadIdx.x >> 5;
                    region_append(keep[c], v[c], st.band_buf + w * BAND_REGION, &st.band_n[w],
                                  BAND_REGION, true, t.bandq, t.band_count, a.n, &ctl->err);
                }
            }
            push_far<SCAN, SPLIT_ILP>(a, st, t, keep, cand, v, [&](int c) { return (uint32_t)d[c]; });
            push_near<SPLIT_ILP>(a, st, t, true, push, v, deg);
        }
        flush_stage(st, t, a.n, &ctl->err);
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) {
            if (first) ctl->exit_reason = 4;
            break;
        }
        n_light = min(ldcg_u32(&ctl->near_count[its % 3]), a.n);
        n_heavy = min(ldcg_u32(&ctl->heavy_count[its % 3]), a.heavy_cap);
        if (first) {
            ctl->pull_hsum = 0;      // read after the pass's barrier, before this one
        }
        it = its;
        cur_dense = dense_out;        // the split set the next frontier's bits
        listed = SCAN && (listed || !step);
        if (it >= a.max_iters) {
            if (first) {
                atomicOr(&ctl->err, ERR_TIMEOUT);
                ctl->exit_reason = 2;
            }
            break;
        }
    }
    // counters
    unsigned long long sum_a = attempts, sum_i = improved;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        sum_a += __shfl_xor_sync(FULL, sum_a, o);
        sum_i += __shfl_xor_sync(FULL, sum_i, o);
    }
    if (lane == 0) {
        atomicAdd(&ctl->relax_attempts, sum_a);
        atomicAdd(&ctl->relax_improved, sum_i);
    }
    if (NARROW && __any_sync(FULL, narrow_miss) && lane == 0) atomicOr(&ctl->err, ERR_NARROW);
    if (first) {
        ctl->iterations = it;
        ctl->phases = phase;
        ctl->bands = bands;
        ctl->end_ns = global_ns();
    }
}
// ---------------------------------------------------------------------------
// export: packed labels -> (cell seed id, distance, predecessor id)
// ---------------------------------------------------------------------------

__global__ void export_kernel(uint32_t n, const uint2 *__restrict__ adj,
                              const uint2 *__restrict__ adj_near, uint32_t near,
                              const uint64_t *__restrict__ label,
                              const uint32_t *__restrict__ label32, uint32_t lshift,
                              const uint32_t *__restrict__ pred_arc,
                              const int32_t *__restrict__ seeds,
                              const uint32_t *__restrict__ orig_of, int32_t *cell, uint32_t *dist,
                              int32_t *pred) {
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const uint32_t v = caller_id(orig_of, u);       // outputs are in the caller's ids
        uint64_t lab = label32 ? widen_label(label32[u], lshift) : label[u];
        if (lab == INF64) {
            if (cell) cell[v] = -1;
            if (dist) dist[v] = INF32;
            if (pred) pred[v] = -1;
            continue;
        }
        if (cell) cell[v] = seeds[(uint32_t)lab];
        if (dist) dist[v] = (uint32_t)(lab >> 32);
        if (pred) {
            uint32_t pa = pred_arc[u];
            // (the near vertices' arcs are indices in the split rows)
            pred[v] = pa == SEED_ARC ? (int32_t)v
                      : pa == INF32 ? -1
                      : (int32_t)caller_id(orig_of, (label32 && label32[u] < near ? adj_near : adj)[pa].x);
        }
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

static int grid_for(uint64_t items, int threads) {
    uint64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    const uint64_t cap = (uint64_t)current_sm_count() * 16;
    if (b > cap) b = cap;
    return (int)b;
}

cudaError_t launch_init(const DevGraph &g, Workspace &ws, uint32_t k, uint32_t delta,
                        cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(ws.ctl, 0, sizeof(Control), s);
    if (e != cudaSuccess) return e;
    uint32_t *l32 = ws.narrow ? ws.label32 : nullptr;
    init_labels_kernel<<<grid_for(g.n, 256), 256, 0, s>>>(g.n, ws.label, l32, ws.pred_arc);
    init_seeds_kernel<<<(k + 255) / 256, 256, 0, s>>>(g.row_ptr, active_lend(g, delta), ws.seeds,
                                                       g.new_of, k, ws.label, l32,
                                                       ws.pred_arc, ws.stamp_near,
                                                       ws.epoch_near, ws.q[0], ws.hq[0],
                                                       g.heavy_chunk_cap, g.n, ws.ctl);
    return cudaGetLastError();
}

// Co-resident blocks per SM that every form of the kernel reaches.
int sssp_occupancy(int threads) {
    const void *forms[] = {(const void *)sssp_kernel<false, false, SSSP_BLOCKS>,
                           (const void *)sssp_kernel<false, true, SSSP_BLOCKS>,
                           (const void *)sssp_kernel<true, false, SSSP_BLOCKS>,
                           (const void *)sssp_kernel<true, true, SSSP_BLOCKS>};
    int least = 0;
    for (const void *fn : forms) {
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, 0) != cudaSuccess) return 0;
        least = least ? (n < least ? n : least) : n;
        if (least < 1) return 0;
    }
    return least;
}

cudaError_t launch_sssp(const DevGraph &g, Workspace &ws, const Geometry &geo,
                        const SsspParams &p, cudaStream_t s) {
    SsspArgs a;
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.n = g.n;
    a.label = ws.label;
    a.label32 = ws.label32;
    a.lshift = ws.lshift;
    a.lstep = 1u << ws.lshift;
    a.lmiss = (1ull << 32) - a.lstep;        // distances up to 2^(32 - rank bits) - 2 fit
    a.stamp_near = ws.stamp_near;
    a.stamp_far = ws.stamp_far;
    a.q0 = ws.q[0];
    a.q1 = ws.q[1];
    a.hq0 = ws.hq[0];
    a.hq1 = ws.hq[1];
    a.far0 = ws.far[0];
    a.far1 = ws.far[1];
    a.ctl = ws.ctl;
    a.delta = p.delta;
    a.max_iters = p.max_iters;
    a.base_near = p.base_near;
    a.base_far = p.base_far;
    a.heavy_cap = g.heavy_chunk_cap;
    a.local_rounds = p.local_rounds;
    a.stamp_band = ws.stamp_band;
    a.band_q = ws.band_q;
    a.band_hq = ws.band_hq;
    a.base_band = p.base_band;
    a.defer = p.delta <= g.max_w ? 1u : 0u;
    a.trace = p.trace;
    a.dense = p.dense;
    a.pull = p.far_scan ? p.pull : 0u;
    a.tail = p.tail;
    a.m = g.m;
    a.step0 = p.far_scan ? first_step(p.delta, g.delta0, g.max_w, g.even) : 0u;
    // Two blocks per SM spill little or nothing (see SSSP_BLOCKS) and go faster
    // through the chain of loads of a hop, three keep more arcs in flight.  Two, of
    // three: R-MAT 12 0.224 ms of 0.257, 10^6 vertices (k = 101) 1.04 of 1.07,
    // R-MAT 22 (k = 64) 1.50 of 1.58; grid 1021 x 733 1.85 of 1.96, 2048 x 1900
    // 10.4 of 11.1.  Three, of two: R-MAT 24 5.6 ms of 6.2, R-MAT 26 (degree 8)
    // 7.9 of 8.1; with local rounds asked for, where every warp has a chain of
    // its own, grid 4096 x 4096 7.8 of 8.05.
    const bool two = p.far_scan ? g.m < 1ull << 28 : !p.local_rounds;
    const int blocks = two ? std::min(geo.sssp_blocks, 2 * geo.sm_count) : geo.sssp_blocks;
    // Thin frontiers with the far pile (see the kernel).  Few arcs per vertex
    // mean a high diameter (grids, paths, trees): below eight vertices per
    // warp a frontier there also takes 16 warp-local rounds, so that a
    // barrier is paid every 16 hops, until one has more than a batch to relax
    // (grid 1021 x 733, k = 37, three blocks per SM: 1.98 ms; 2.39 without that
    // limit; split early without rounds 4.9, neither 6.7; 300 x 333, k = 200: 0.58 against 1.21).
    // On denser graphs a warp's own rounds would relax hub rows alone (R-MAT
    // 12: 0.93 ms against 0.20); there a frontier below one vertex per warp
    // only splits early (0.29 against 0.31 ms).  With local rounds asked for
    // the same lines hold for the early split (grid 4096 x 4096: 7.8 ms; 8.1
    // without, 7.9 at one vertex per warp, 8.2 at 32).
    const uint32_t warps = (uint32_t)(blocks * (geo.threads / 32));
    const bool sparse_rows = g.m <= 8ull * g.n;
    a.thin = sparse_rows ? 8 * warps : warps;
    a.thin_rounds = sparse_rows ? 16u : 0u;
    a.n_big = g.n_big;
    a.n_live = g.n_live;
    a.n_words = (g.n + 31) / 32;
    a.nbm0 = ws.nbm[0];
    a.nbm1 = ws.nbm[1];
    a.bbm = ws.bbm;
    a.items = g.items;
    a.sparse_items = g.sparse_items;
    a.n_items = g.n_items;
    a.n_sparse_items = g.n_sparse_items;
    a.lend = active_lend(g, p.delta);
    if (a.lend) a.adj = g.adj_w;        // rows partitioned by weight class
    void *args[] = {&a};
    auto form = [&](auto b) {
        constexpr int B = decltype(b)::value;
        return ws.narrow ? (p.far_scan ? (const void *)sssp_kernel<true, true, B>
                                       : (const void *)sssp_kernel<true, false, B>)
                         : (p.far_scan ? (const void *)sssp_kernel<false, true, B>
                                       : (const void *)sssp_kernel<false, false, B>);
    };
    const void *fn = two ? form(std::integral_constant<int, 2>()) : form(std::integral_constant<int, SSSP_BLOCKS>());
    return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(geo.threads), args, 0, s);
}

cudaError_t launch_export(const DevGraph &g, Workspace &ws, uint32_t split_delta, int32_t *cell,
                          uint32_t *dist, int32_t *pred, cudaStream_t s) {
    export_kernel<<<grid_for(g.n, 256), 256, 0, s>>>(
        g.n, g.adj, g.adj_w, split_delta ? near_label(ws, split_delta) : 0u, ws.label,
        ws.narrow ? ws.label32 : nullptr, ws.lshift, ws.pred_arc, ws.seeds, g.orig_of, cell, dist,
        pred);
    return cudaGetLastError();
}

}  // namespace stn
