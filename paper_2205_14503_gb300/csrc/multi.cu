// Multi-query Voronoi cells and bridge scan (the batched and serving modes).
//
// The arithmetic per query is exactly the single-query path's (Algorithm 2
// Steps 1-2 with the same packed (distance, rank) atomicMin fixed point and
// the same tie rules); what changes is how the work of up to 64 queries is
// shared:
//  * labels are vertex-major, label[v * 64 + q], so relaxing one arc for all
//    pending slots is one contiguous 256-byte run of atomics; a label is 32
//    bits, (distance << b) | rank with b the bits of the slot's largest rank
//    (ordered by (distance, rank) as the 64-bit form), and a slot whose
//    distances do not fit is answered by the single-query path instead;
//  * a frontier entry is a vertex; nmask[v] says which slots must relax
//    v's arcs, so a CSR row is read once for all of them;
//  * each slot has its own near/far threshold T[q] and far accounting, so a
//    slot admitted mid-run starts its own bands (continuous batching);
//  * the persistent kernel can yield at an iteration boundary (a slot
//    converged, or the host rang the doorbell), keeping all state in device
//    memory, and resume later with more slots;
//  * light and heavy arcs are split per slot as in the single-query kernel:
//    while a slot's band iterates only arcs lighter than delta are relaxed,
//    a per-vertex mask records which slots relaxed the vertex in their
//    current band (vertices with any bit set are kept in a band list), and
//    when a slot's near work drains its heavy arcs are relaxed once, in the
//    next shared iteration, for the listed vertices with its bit;
//  * a slot whose band holds most of the graph (its first one as a rule, its
//    second at the latest) runs the heavy-arc pass in the pull form and
//    finishes as one unbounded band over whole rows (its tail), as in the
//    single-query kernel.
#include "multi.h"

namespace stn {

// (arc, slot) pairs in flight per lane, and blocks per SM: R-MAT 22, 64 queries,
// Voronoi part 26 ms at two and six (24 with the chunks on demand), 28 and 31 at
// two and five or four, 32 at four and five.
constexpr int MQ_ILP = 2;
constexpr int MQ_BLOCKS = 6;
// The last MQ_TAKE of every 32 chunks of the pair pass go to whichever warp is
// free: the wait at the end of an iteration, up to 0.3 ms of 3, came from warps
// whose chunks had many improving pairs.  R-MAT 22, 64 queries: waits 5.3 ->
// 1.9 ms, batch 46.3 -> 44.3 ms (46.5 -> 45.5 at 4 of 32, the same at 16).
// Chunks of less than MQ_TAKE_PAIRS pairs are left with their warps: there the
// search for a chunk costs as much as its pairs.
constexpr uint32_t MQ_TAKE = 8;
constexpr uint64_t MQ_TAKE_PAIRS = 64;
constexpr uint32_t MQ_HOLD = 16;   // iterations a drained first band waits for others
constexpr uint32_t MQ_NEAR_STAGE = 1024;
constexpr uint32_t MQ_FAR_STAGE = 512;

struct MqArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;
    uint32_t n;
    uint32_t *label;
    unsigned long long *nmask, *fmask;
    uint32_t *stamp_near, *in_far;
    uint32_t *q0, *q1;
    unsigned long long *item_mask;   // per frontier item: the slots it relaxes
    uint64_t *item_pre;              // per item: (arc, slot) pairs before it in its block segment
    uint64_t *bsum;                  // per block: pairs in its segment
    uint32_t *far0, *far1;
    unsigned long long *bmask;       // per vertex: slots that relaxed it in their current band
    uint32_t *bl0, *bl1, *bl2;       // band lists
    MqControl *ctl;
    const uint32_t *doorbell;
    uint32_t delta;
    uint32_t base_near;
    uint32_t max_iters;
    uint32_t yield;          // leave once this many slots converged (0: only when all did)
    uint32_t defer;          // light/heavy arc split on (some weight >= delta)
    // with the split: end of each row's light part in the weight-partitioned
    // adjacency `adj` (null: rows are unpartitioned and arcs are filtered)
    const uint32_t *lend;
    uint32_t pull;           // a slot whose band holds most of the graph takes the pull form and the tail
    const uint64_t *__restrict__ heavy_chunks;   // hub rows in CHUNK-arc pieces
    uint32_t n_heavy_chunks;
};

__device__ __forceinline__ uint32_t *band_list(const MqArgs &a, uint32_t i) {
    return i == 0 ? a.bl0 : (i == 1 ? a.bl1 : a.bl2);
}

constexpr int MQ_WARPS = 256 / 32;
constexpr int MQ_MAX_BLOCKS = 1024;

struct MqTargets {
    uint32_t *qn, *qn_count;
    unsigned long long *act;
    uint32_t *farq, *far_count;
    uint32_t *fmin;          // ctl->fmin[pile]
    uint32_t tag_next;
};

struct MqStage {
    uint64_t boff[MQ_MAX_BLOCKS];          // pair offset of each block's frontier segment
    uint64_t wtot[MQ_WARPS];
    uint64_t carry, W;
    uint32_t near_buf[MQ_NEAR_STAGE];
    uint32_t far_buf[MQ_FAR_STAGE];
    uint32_t near_n, far_n, base_near, base_far;
    unsigned long long act;
    unsigned long long T[MQ_SLOTS];        // current thresholds (block copy)
    unsigned long long Tnew[MQ_SLOTS];     // thresholds after a split
    uint32_t fmin[MQ_SLOTS];               // far-distance minimum of this segment
    int32_t fpend[MQ_SLOTS];               // change of far_pending in this segment
    unsigned long long mag[MQ_SLOTS + 1];  // ceil(2^40 / c) for c = 2..64 (divmod by c)
    uint32_t lshift[MQ_SLOTS];             // rank bits of each slot's labels
    uint32_t cov[MQ_SLOTS];                // sampled arcs with a settled end, then the grid's sum
    MqTargets t;                           // where this iteration's pushes go
    unsigned long long miss;               // slots whose distances left the 32-bit labels
    // each warp's window of work items in the pair pass: {vertex, first arc,
    // first pair, end of pairs}, {first arc index, last arc index, slot mask},
    // slots | (window flags)
    uint4 wa[MQ_WARPS][32], wb[MQ_WARPS][32];
    uint32_t wc[MQ_WARPS][32];
};

// Slot q's label of v in the 64-bit form (dist << 32) | rank.
__device__ __forceinline__ uint64_t mq_label(const uint32_t *label, uint64_t v, uint32_t q,
                                             uint32_t shift) {
    return widen_label(ldcg_u32(&label[v * MQ_SLOTS + q]), shift);
}

__device__ __forceinline__ int popc64(unsigned long long x) { return __popcll(x); }

// Inclusive scan of one 64-bit value per thread over a 256-thread block;
// wtot[] receives the per-warp inclusive totals (wtot[MQ_WARPS-1] = block
// total after the call).  Every thread of the block must call it.
__device__ __forceinline__ uint64_t block_inclusive_scan64(uint64_t x, uint64_t *wtot) {
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint64_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) wtot[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t acc = 0;
        for (int i = 0; i < MQ_WARPS; ++i) {
            acc += wtot[i];
            wtot[i] = acc;
        }
    }
    __syncthreads();
    return x + (w ? wtot[w - 1] : 0);
}

__device__ __forceinline__ uint32_t nth_bit64(unsigned long long m, uint32_t t) {
    uint32_t lo = (uint32_t)m, pl = (uint32_t)__popc(lo);
    return t < pl ? nth_set_bit(lo, t) : 32 + nth_set_bit((uint32_t)(m >> 32), t - pl);
}

__device__ __forceinline__ unsigned long long warp_or64(unsigned long long x) {
    uint32_t lo = __reduce_or_sync(FULL, (uint32_t)x);
    uint32_t hi = __reduce_or_sync(FULL, (uint32_t)(x >> 32));
    return ((unsigned long long)hi << 32) | lo;
}

__device__ __forceinline__ void seg_reset(MqStage &st) {
    if (threadIdx.x == 0) {
        st.near_n = 0;
        st.far_n = 0;
        st.act = 0;
    }
    if (threadIdx.x < MQ_SLOTS) {
        st.fmin[threadIdx.x] = INF32;
        st.fpend[threadIdx.x] = 0;
    }
    __syncthreads();
}

__device__ __forceinline__ void seg_flush(MqStage &st, const MqTargets &t, MqControl *ctl,
                                          uint32_t n) {
    __syncthreads();
    uint32_t nn = min(st.near_n, MQ_NEAR_STAGE), nf = min(st.far_n, MQ_FAR_STAGE);
    if (threadIdx.x == 0) {
        st.base_near = nn ? atomicAdd(t.qn_count, nn) : 0;
        st.base_far = nf ? atomicAdd(t.far_count, nf) : 0;
        if (st.act) atomicOr(t.act, st.act);
    }
    if (threadIdx.x < MQ_SLOTS) {
        uint32_t q = threadIdx.x;
        if (st.fmin[q] != INF32) atomicMin(&t.fmin[q], st.fmin[q]);
        if (st.fpend[q]) atomicAdd(&ctl->far_pending[q], st.fpend[q]);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nn; i += blockDim.x) {
        uint32_t slot = st.base_near + i;
        if (slot < n) t.qn[slot] = st.near_buf[i];
        else atomicOr(&ctl->err, ERR_CAPACITY);
    }
    for (uint32_t i = threadIdx.x; i < nf; i += blockDim.x) {
        uint32_t slot = st.base_far + i;
        if (slot < n) t.farq[slot] = st.far_buf[i];
        else atomicOr(&ctl->err, ERR_CAPACITY);
    }
}

// A vertex with near work joins the next frontier through the staging
// buffer.  (Hubs need no special handling: work is split by pairs.)
__device__ __forceinline__ void mq_push_near(const MqArgs &a, MqStage &st, const MqTargets &t,
                                             bool want, uint32_t v) {
    stage_append(want, v, st.near_buf, &st.near_n, MQ_NEAR_STAGE, t.qn, t.qn_count, a.n,
                 &a.ctl->err);
}

// One slot served by a lane: its number, its label's rank bits and the label
// (as stored) of the vertex being relaxed.
struct MqLane {
    uint32_t q, sh, lab;
    uint32_t room, whi;      // arcs of weight `room` on do not fit; from `whi` on are not relaxed
};

// Sums of label and weight step at or above this do not fit slot labels of
// `sh` rank bits.
__device__ __forceinline__ uint64_t mq_label_limit(uint32_t sh) { return (1ull << 32) - (1ull << sh); }

// The smallest label of a distance at or above T (saturating).
__device__ __forceinline__ uint32_t mq_threshold_label(unsigned long long T, uint32_t sh) {
    return T >= (1ull << (32 - sh)) ? INF32 : (uint32_t)T << sh;
}

// Relaxes up to MQ_ILP (arc, slot) pairs per lane: arc record e[i] (weight 0:
// no pair) for the lane's slot s0, or with TWO slots per lane s0 and s1 in
// turn.  Only arcs of weight in [wlo, the lane's whi) are relaxed.  Labels are
// compared and sent as stored: lab + (weight << rank bits), which fits for
// weights below the lane's room.  UNIFORM: at every i all lanes have the same
// arc, so the masks and the stamp of its head take one atomic for the warp.
template <bool TWO, bool UNIFORM>
__device__ __forceinline__ void mq_relax(const MqArgs &a, MqStage &st, const MqTargets &t,
                                         const uint2 (&e)[MQ_ILP], const MqLane &s0,
                                         const MqLane &s1, uint32_t wlo, uint32_t &attempts,
                                         uint32_t &improved) {
    uint32_t nl[MQ_ILP], cur[MQ_ILP];
#pragma unroll
    for (int i = 0; i < MQ_ILP; ++i) {
        const MqLane &s = TWO && (i & 1) ? s1 : s0;
        nl[i] = INF32;
        cur[i] = 0;
        if (e[i].y < wlo || e[i].y >= s.whi) continue;
        ++attempts;
        if (e[i].y >= s.room) {
            atomicOr(&st.miss, 1ull << s.q);     // the slot is answered by the single-query path
        } else {
            // read first: most proposals do not improve, and a load costs far
            // less L2 throughput than an atomic
            nl[i] = s.lab + (e[i].y << s.sh);
            cur[i] = ldcg_u32(&a.label[(uint64_t)e[i].x * MQ_SLOTS + s.q]);
        }
    }
    bool imp[MQ_ILP], any_imp = false;
#pragma unroll
    for (int i = 0; i < MQ_ILP; ++i) {
        const MqLane &s = TWO && (i & 1) ? s1 : s0;
        imp[i] = nl[i] < cur[i] &&
                 nl[i] < atomicMin(&a.label[(uint64_t)e[i].x * MQ_SLOTS + s.q], nl[i]);
        any_imp |= imp[i];
    }
    // most rounds improve nothing: skip the append machinery then
    if (!__any_sync(FULL, any_imp)) return;
    bool to_near[MQ_ILP], to_far[MQ_ILP];
    unsigned long long act = 0;
#pragma unroll
    for (int i = 0; i < MQ_ILP; ++i) {
        const MqLane &s = TWO && (i & 1) ? s1 : s0;
        to_near[i] = to_far[i] = false;
        const uint32_t v = e[i].x;
        const unsigned long long bit = 1ull << s.q;
        const bool near = imp[i] && (nl[i] >> s.sh) < st.T[s.q], far = imp[i] && !near;
        if (imp[i]) ++improved;
        if (near) act |= bit;
        if (UNIFORM) {
            if (!__any_sync(FULL, imp[i])) continue;
            const unsigned long long nb = warp_or64(near ? bit : 0ull);
            const unsigned long long fb = warp_or64(far ? bit : 0ull);
            // the lowest lane with an improvement speaks for the warp
            const uint32_t lead = __ffs(__ballot_sync(FULL, imp[i])) - 1;
            unsigned long long old = 0;
            if (lane_id() == lead) {
                if (nb) {
                    atomicOr(&a.nmask[v], nb);
                    to_near[i] = atomicExch(&a.stamp_near[v], t.tag_next) != t.tag_next;
                }
                if (fb) {
                    old = atomicOr(&a.fmask[v], fb);
                    to_far[i] = atomicExch(&a.in_far[v], 1u) == 0;
                }
            }
            if (fb) {
                old = __shfl_sync(FULL, old, lead);
                if (far) {
                    if (!(old & bit)) atomicAdd(&st.fpend[s.q], 1);
                    atomicMin(&st.fmin[s.q], nl[i] >> s.sh);
                }
            }
        } else if (near) {
            atomicOr(&a.nmask[v], bit);
            to_near[i] = atomicExch(&a.stamp_near[v], t.tag_next) != t.tag_next;
        } else if (far) {
            const unsigned long long old = atomicOr(&a.fmask[v], bit);
            if (!(old & bit)) atomicAdd(&st.fpend[s.q], 1);
            atomicMin(&st.fmin[s.q], nl[i] >> s.sh);
            to_far[i] = atomicExch(&a.in_far[v], 1u) == 0;
        }
    }
    act = warp_or64(act);
    if (lane_id() == 0 && act) atomicOr(&st.act, act);
#pragma unroll
    for (int i = 0; i < MQ_ILP; ++i) {
        mq_push_near(a, st, t, to_near[i], e[i].x);
        stage_append(to_far[i], e[i].x, st.far_buf, &st.far_n, MQ_FAR_STAGE, t.farq, t.far_count,
                     a.n, &a.ctl->err);
    }
}

// Pull form of the heavy-arc pass of the slots in P.  A slot in its first band
// has threshold delta; once its near work drained, every label below it is
// final, and a heavy arc (weight delta or more) brings a vertex still at or
// above it only a proposal at or above it.  (In a second band the same holds
// for the band's vertices, and the first band's heavy arcs have been pushed.)  So instead of
// pushing the heavy arcs of the band's vertices, every vertex unsettled in
// some slot of P reads its own heavy arcs and, per arc, the label run of the
// other end.  Lane l serves slots 2l and 2l + 1 (one 8-byte load of a run per
// arc), keeps their best proposals from settled ends in registers and, after
// the row, sends one atomicMin per improved (vertex, slot) and does the
// bookkeeping of mq_relax for it (a far proposal: far mask, far pending
// count, far minimum, far pile).  No frontier or band item relaxes those
// slots in the iteration: the band items leave out the slots of P, and those
// slots have no near work.
// What bounds it: the latency of the label runs, so PULL_ARCS of them are in
// flight per warp (the arc records come 32 at a time, a lane each), and hub
// rows are cut in pieces over the grid: one arc after another, a hub left
// unsettled in some slot held up the whole sweep (R-MAT 22, 64 queries: the
// batch took 100 or 205 ms, by whether the draw of seeds left one).  With one
// shared sweep and the tails behind it the same batch took 51 ms: Voronoi
// part 70 -> 31 ms, 66 -> 23 iterations, 6 -> 1 sweeps.
constexpr int PULL_ARCS = 4;
constexpr int PULL_ROWS = 4;       // vertices whose labels are loaded together

__device__ __forceinline__ void mq_pull_row(const MqArgs &a, MqStage &st, const MqTargets &t,
                                            uint32_t v, uint32_t s, uint32_t r1, uint2 mine,
                                            uint2 lv, bool ua,
                                            bool ub, uint32_t sha, uint32_t shb, uint32_t Ta,
                                            uint32_t Tb, uint32_t &attempts, uint32_t &improved) {
    const uint32_t lane = lane_id(), qa = 2 * lane, qb = qa + 1;
    uint32_t ba = INF32, bb = INF32;
    for (uint32_t w0 = s, cnt; w0 != r1; w0 += cnt) {        // (r1 + 31 may wrap)
        cnt = min(32u, r1 - w0);
        if (w0 != s) mine = lane < cnt ? __ldcs(&a.adj[w0 + lane]) : make_uint2(0, 0);
        for (uint32_t i = 0; i < cnt; i += PULL_ARCS) {
            uint2 x[PULL_ARCS];
#pragma unroll
            for (int k = 0; k < PULL_ARCS; ++k) {
                const uint32_t head = __shfl_sync(FULL, mine.x, i + k);
                const uint32_t w = __shfl_sync(FULL, mine.y, i + k);
                x[k] = make_uint2(INF32, INF32);
                if (w >= a.delta && (ua || ub))      // (past the row's end w = 0; light arcs
                                                     // only on unpartitioned rows)
                    x[k] = __ldcg(reinterpret_cast<const uint2 *>(
                        &a.label[(uint64_t)head * MQ_SLOTS + qa]));
            }
#pragma unroll
            for (int k = 0; k < PULL_ARCS; ++k) {
                const uint32_t w = __shfl_sync(FULL, mine.y, i + k);
                if (ua && x[k].x < Ta) {             // a settled end proposes
                    ++attempts;
                    const uint64_t sum = ((uint64_t)w << sha) + x[k].x;
                    if (sum < mq_label_limit(sha)) ba = min(ba, (uint32_t)sum);
                    else if (lv.x == INF32) atomicOr(&st.miss, 1ull << qa);
                }
                if (ub && x[k].y < Tb) {
                    ++attempts;
                    const uint64_t sum = ((uint64_t)w << shb) + x[k].y;
                    if (sum < mq_label_limit(shb)) bb = min(bb, (uint32_t)sum);
                    else if (lv.y == INF32) atomicOr(&st.miss, 1ull << qb);
                }
            }
        }
    }
    uint32_t *dst = &a.label[(uint64_t)v * MQ_SLOTS + qa];
    const bool ia = ua && ba < lv.x && ba < atomicMin(dst, ba);
    const bool ib = ub && bb < lv.y && bb < atomicMin(dst + 1, bb);
    const bool fa = ia && ba >= Ta, fb = ib && bb >= Tb;
    const unsigned long long nbits = warp_or64((ia && !fa ? 1ull << qa : 0ull) | (ib && !fb ? 1ull << qb : 0ull));
    const unsigned long long fbits = warp_or64((fa ? 1ull << qa : 0ull) | (fb ? 1ull << qb : 0ull));
    if (!(nbits | fbits)) return;
    improved += (ia ? 1u : 0u) + (ib ? 1u : 0u);
    unsigned long long fold = 0;
    bool to_far = false, to_near = false;
    if (lane == 0) {
        if (fbits) {
            fold = atomicOr(&a.fmask[v], fbits);
            to_far = atomicExch(&a.in_far[v], 1u) == 0;
        }
        if (nbits) {
            atomicOr(&a.nmask[v], nbits);
            to_near = atomicExch(&a.stamp_near[v], t.tag_next) != t.tag_next;
            atomicOr(&st.act, nbits);
        }
    }
    fold = __shfl_sync(FULL, fold, 0);
    if (fa) {
        if (!((fold >> qa) & 1ull)) atomicAdd(&st.fpend[qa], 1);
        atomicMin(&st.fmin[qa], ba >> sha);
    }
    if (fb) {
        if (!((fold >> qb) & 1ull)) atomicAdd(&st.fpend[qb], 1);
        atomicMin(&st.fmin[qb], bb >> shb);
    }
    mq_push_near(a, st, t, to_near, v);
    stage_append(to_far, v, st.far_buf, &st.far_n, MQ_FAR_STAGE, t.farq, t.far_count, a.n,
                 &a.ctl->err);
}

__device__ __noinline__ void mq_pull_sweep(const MqArgs &a, MqStage &st, unsigned long long P,
                                           uint32_t *qn, uint32_t *qn_count, uint32_t *farq,
                                           uint32_t *far_count, uint32_t tag_next,
                                           uint32_t &attempts, uint32_t &improved) {
    MqTargets t;
    t.qn = qn;
    t.qn_count = qn_count;
    t.act = nullptr;
    t.farq = farq;
    t.far_count = far_count;
    t.fmin = nullptr;
    t.tag_next = tag_next;
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t qa = 2 * lane, qb = qa + 1;
    const uint32_t sha = st.lshift[qa], shb = st.lshift[qb];
    // a slot outside P is settled everywhere: threshold label INF32 + nothing
    const bool pa = (P >> qa) & 1ull, pb = (P >> qb) & 1ull;
    const uint32_t Ta = mq_threshold_label(st.T[qa], sha), Tb = mq_threshold_label(st.T[qb], shb);
    const uint32_t n_items = a.n_heavy_chunks + (a.n + PULL_ROWS - 1) / PULL_ROWS;
    // Row offsets of an item's vertices, one per lane (starts and the last
    // end in lanes 0..PULL_ROWS, starts of the heavy parts from lane 8 on),
    // fetched an item ahead.
    auto offsets = [&](uint32_t wi) {
        if (wi >= n_items) return 0u;
        const uint32_t v0 = wi < a.n_heavy_chunks ? (uint32_t)(a.heavy_chunks[wi] >> 32)
                                                  : (wi - a.n_heavy_chunks) * PULL_ROWS;
        const uint32_t r = lane & 7u, v = min(v0 + r, a.n);
        if (lane < 8) return r <= PULL_ROWS ? a.row_ptr[v] : 0u;
        if (lane >= 16 || r >= PULL_ROWS || v >= a.n) return 0u;
        return a.lend ? a.lend[v] : a.row_ptr[v];
    };
    uint32_t next = offsets(warp);
    for (uint32_t wi = warp; wi < n_items; wi += nwarps) {
        const uint32_t off = next;
        next = offsets(wi + nwarps);
        const bool hub = wi < a.n_heavy_chunks;
        uint32_t v0, c = 0, rows = 1;
        if (hub) {
            const uint64_t item = a.heavy_chunks[wi];
            v0 = (uint32_t)(item >> 32);
            c = (uint32_t)item;
        } else {
            v0 = (wi - a.n_heavy_chunks) * PULL_ROWS;
            rows = min((uint32_t)PULL_ROWS, a.n - v0);
        }
        // rows without heavy arcs (isolated vertices above all) need no look
        // at their labels; hub rows are covered by their pieces
        uint32_t s[PULL_ROWS], e[PULL_ROWS];
        uint2 lv[PULL_ROWS], mine[PULL_ROWS];
#pragma unroll
        for (int r = 0; r < PULL_ROWS; ++r) {
            const uint32_t r0 = __shfl_sync(FULL, off, r);
            e[r] = __shfl_sync(FULL, off, r + 1);
            s[r] = __shfl_sync(FULL, off, 8 + r);
            if (hub) {
                const RowPiece p = row_piece(s[r], e[r], c * CHUNK, r == 0 ? CHUNK : 0u);
                s[r] = p.first;
                e[r] = p.first + p.count;
            } else if ((uint32_t)r >= rows || e[r] - r0 >= HEAVY_DEG) {
                e[r] = s[r];
            }
            lv[r] = make_uint2(0, 0);
            if (e[r] > s[r] && (pa || pb))
                lv[r] = __ldcg(reinterpret_cast<const uint2 *>(&a.label[(uint64_t)(v0 + r) * MQ_SLOTS + qa]));
        }
        bool ua[PULL_ROWS], ub[PULL_ROWS];
#pragma unroll
        for (int r = 0; r < PULL_ROWS; ++r) {
            ua[r] = e[r] > s[r] && pa && lv[r].x >= Ta;
            ub[r] = e[r] > s[r] && pb && lv[r].y >= Tb;
            mine[r] = make_uint2(0, 0);
            if (!__any_sync(FULL, ua[r] || ub[r])) e[r] = s[r];
            else if (lane < e[r] - s[r]) mine[r] = __ldcs(&a.adj[s[r] + lane]);
        }
#pragma unroll
        for (int r = 0; r < PULL_ROWS; ++r)
            if (e[r] > s[r])
                mq_pull_row(a, st, t, v0 + r, s[r], e[r], mine[r], lv[r], ua[r], ub[r], sha, shb,
                            Ta, Tb, attempts, improved);
    }
}

// Which of the slots in `ask` have settled most arcs' ends, by a sample of one
// arc per warp, spread evenly over the arcs (a slot asks only if some arc
// weighs delta or more, so there are arcs).  One grid barrier; all blocks get
// the same answer.  A failed barrier sets `reason`.
// Why the pull form and the tail wait for that: they pay where little of the
// graph is left.  A slot whose seeds lie off the core settled next to nothing
// in its first band, made the sweep read every row (2.4 -> 9.6 ms) and then
// carried the whole graph through its tail, alone in its label runs.  Such a
// slot has its heavy arcs pushed instead and gets a second band, once (its
// threshold starts at the nearest vertex it left out).  R-MAT 22, 64 queries,
// draws with one to five such slots: 61-72 -> 44-51 ms, the others the same
// (44-47); each ask costs 20 us.
__device__ __noinline__ unsigned long long mq_wide_bands(const MqArgs &a, MqStage &st,
                                                         unsigned long long ask, uint32_t &bar_target,
                                                         uint32_t &reason) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    MqControl *ctl = a.ctl;
    if (threadIdx.x < MQ_SLOTS) st.cov[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t arcs = a.row_ptr[a.n];
    const uint32_t v = a.adj[(uint64_t)arcs * warp / nwarps].x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t q = lane + 32 * h;
        if (((ask >> q) & 1ull) &&
            ldcg_u32(&a.label[(uint64_t)v * MQ_SLOTS + q]) < mq_threshold_label(st.T[q], st.lshift[q]))
            atomicAdd(&st.cov[q], 1u);
    }
    __syncthreads();
    if (threadIdx.x < MQ_SLOTS && st.cov[threadIdx.x]) atomicAdd(&ctl->cov[threadIdx.x], st.cov[threadIdx.x]);
    if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) { reason = 5; return 0ull; }
    if (threadIdx.x < MQ_SLOTS) st.cov[threadIdx.x] = ldcg_u32(&ctl->cov[threadIdx.x]);
    __syncthreads();
    const uint32_t lo = __ballot_sync(FULL, 2 * st.cov[lane] >= nwarps);
    const uint32_t hi = __ballot_sync(FULL, 2 * st.cov[lane + 32] >= nwarps);
    return (((unsigned long long)hi << 32) | lo) & ask;
}

__global__ void __launch_bounds__(256, MQ_BLOCKS) mq_sssp_kernel(const __grid_constant__ MqArgs a) {
    __shared__ MqStage st;
    MqControl *ctl = a.ctl;
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const bool first = gtid == 0;
    uint32_t attempts = 0, improved = 0;     // this thread's
    uint32_t it = ldcg_u32(&ctl->it), fc = ldcg_u32(&ctl->fc);
    unsigned long long infl = __ldcg(&ctl->inflight) & ~__ldcg(&ctl->converged);
    unsigned long long conv_total = 0;
    // heavy-arc passes: H = slots whose pass runs in this iteration
    unsigned long long H = __ldcg(&ctl->hpass) & infl;
    unsigned long long hp_done = __ldcg(&ctl->hp_done);
    unsigned long long band0 = __ldcg(&ctl->band0);
    unsigned long long wide = __ldcg(&ctl->wide);       // slots whose band holds most arcs
    unsigned long long late = __ldcg(&ctl->late);       // slots with a narrow band behind them
    unsigned long long tails = __ldcg(&ctl->tails);     // slots in their unbounded tail
    uint32_t held = ldcg_u32(&ctl->held);               // iterations that drained slots waited
    uint32_t pull_sweeps = 0;
    uint32_t bc = ldcg_u32(&ctl->blist);
    if (threadIdx.x < MQ_SLOTS) {
        st.T[threadIdx.x] = __ldcg(&ctl->T[threadIdx.x]);
        st.lshift[threadIdx.x] = ldcg_u32(&ctl->lshift[threadIdx.x]);
    }
    if (threadIdx.x == 0) st.miss = 0;
    if (threadIdx.x <= MQ_SLOTS) {
        const uint32_t c = threadIdx.x;
        st.mag[c] = c > 1 ? ((1ull << 40) + c - 1) / c : 0ull;
    }
    __syncthreads();
    uint32_t iters = 0, reason = 0;
    uint32_t bar_target = 0;

    while (infl) {
        const uint32_t cs = it % 3, ns = (it + 1) % 3;
        const bool odd = it & 1;
        const uint32_t n_items = min(ldcg_u32(&ctl->near_count[cs]), a.n);
        // Work items: the near frontier, then (when some slots run their
        // heavy-arc pass) the band list.  A pass reads list bc and moves the
        // survivors, with this iteration's new listings, to list bc + 1;
        // list bc + 2 (read by the previous pass) is cleared for the next.
        // slots of H whose band holds most of the graph (or their second band)
        // run the pass in the pull form
        const unsigned long long P = a.pull ? (H & band0 & wide) : 0ull;
        const uint32_t n_band = H ? min(ldcg_u32(&ctl->bcount[bc]), a.n) : 0u;
        const uint32_t n_all = n_items + n_band;
        const uint32_t tgt = H ? (bc + 1) % 3 : bc;
        const uint32_t *blo = band_list(a, bc);
        uint32_t *bln = band_list(a, tgt);
        if (first) {
            uint32_t r = (it + 2) % 3;
            ctl->near_count[r] = 0;
            ctl->act[r] = 0;
            ctl->take[r] = 0;
            if (H) ctl->bcount[(bc + 2) % 3] = 0;
        }
        const uint32_t *qc = odd ? a.q1 : a.q0;

        unsigned long long tm0 = first ? global_ns() : 0;
        // Phase A: every frontier vertex takes its pending slot mask; its
        // work is deg x |mask| (arc, slot) pairs; prefix sums per block
        // segment of the frontier.
        const uint32_t seg = (n_all + gridDim.x - 1) / gridDim.x;
        const uint32_t seg_lo = min(n_all, blockIdx.x * seg);
        const uint32_t seg_hi = min(n_all, seg_lo + seg);
        if (threadIdx.x == 0) st.carry = 0;
        __syncthreads();
        for (uint32_t b0 = seg_lo; b0 < seg_hi; b0 += blockDim.x) {
            uint32_t i = b0 + threadIdx.x;
            uint64_t w = 0;
            bool listed = false;
            uint32_t u = 0;
            if (i < seg_hi) {
                unsigned long long M;
                if (i < n_items) {
                    u = ldcg_u32(&qc[i]);
                    M = atomicExch(&a.nmask[u], 0ull);
                    // first slot to relax u in its band lists u
                    if (a.defer && (M & ~tails)) listed = atomicOr(&a.bmask[u], M & ~tails) == 0ull;
                } else {
                    u = ldcg_u32(&blo[i - n_items]);
                    const unsigned long long old = atomicAnd(&a.bmask[u], ~H);
                    M = old & H & ~P;            // the slots whose band closes now (pushed)
                    listed = (old & ~H) != 0ull; // still in other slots' bands
                }
                a.item_mask[i] = M;
                // frontier items relax the light part (the whole row for a
                // slot in its tail, and then for the item's other slots too:
                // relaxing an arc early does no harm), band items the heavy one
                const uint32_t r0 = a.row_ptr[u], r1 = a.row_ptr[u + 1];
                const uint32_t le = a.lend && !(M & tails) ? a.lend[u] : r1;
                const uint32_t deg = i < n_items ? le - r0 : (a.lend ? r1 - le : r1 - r0);
                w = (uint64_t)deg * (uint64_t)popc64(M);
            }
            const uint32_t ls = warp_append(listed, &ctl->bcount[tgt], a.n, &ctl->err);
            if (ls != INF32) bln[ls] = u;
            uint64_t incl = block_inclusive_scan64(w, st.wtot);
            if (i < seg_hi) a.item_pre[i] = st.carry + incl - w;
            __syncthreads();
            if (threadIdx.x == blockDim.x - 1) st.carry += incl;
            __syncthreads();
        }
        if (threadIdx.x == 0) a.bsum[blockIdx.x] = st.carry;
        unsigned long long tm1 = first ? global_ns() : 0;
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) { reason = 5; break; }
        unsigned long long tm2 = first ? global_ns() : 0;
        if (blockIdx.x == 0 && threadIdx.x < MQ_SLOTS) ctl->cov[threadIdx.x] = 0;
        // block offsets and the total
        {
            uint64_t carry = 0;
            for (uint32_t b0 = 0; b0 < gridDim.x; b0 += blockDim.x) {
                uint32_t b = b0 + threadIdx.x;
                uint64_t x = b < gridDim.x ? __ldcg(reinterpret_cast<const unsigned long long *>(&a.bsum[b])) : 0;
                uint64_t incl = block_inclusive_scan64(x, st.wtot);
                if (b < gridDim.x) st.boff[b] = carry + incl - x;
                __syncthreads();
                carry += st.wtot[MQ_WARPS - 1];
                __syncthreads();
            }
            if (threadIdx.x == 0) st.W = carry;
            __syncthreads();
        }
        seg_reset(st);
        MqTargets &t = st.t;
        if (threadIdx.x == 0) {
            t.qn = odd ? a.q0 : a.q1;
            t.qn_count = &ctl->near_count[ns];
            t.act = &ctl->act[ns];
            t.farq = fc ? a.far1 : a.far0;
            t.far_count = &ctl->far_count[fc];
            t.fmin = ctl->fmin[fc];
            t.tag_next = a.base_near + it + 1;
        }
        __syncthreads();

        // Phase B: the W (arc, slot) pairs, numbered arc-major inside each
        // item (arc j, slot t -> j * |mask| + t), are cut into 32 chunks per
        // warp, and warp w takes chunks w, w + nw, w + 2 nw, ... spread over
        // the whole pair space, so a costly region (many improving pairs) is
        // shared by many warps.  Lane i finds the first item of the warp's
        // i-th chunk (all 32 searches at once).  Inside a chunk the warp
        // slides a window of 32 consecutive items (one per lane, loaded in
        // parallel) and spreads the window's pairs over its lanes, MQ_ILP per
        // lane in flight.
        // Registers bound it: six blocks per SM leave 40 per thread, and with
        // the window in registers (eight a lane, read by shuffles), pointers
        // to the push targets and 64-bit label sums a third of the L2 traffic
        // was spilled registers.  So each lane works out its own item's pair
        // range and leaves it in shared memory, the targets are in shared
        // memory too, and a lane compares an arc's weight with the room its
        // label leaves.  R-MAT 22, 64 queries: Voronoi part 31 -> 26 ms (five
        // blocks with more registers 28, four 31).
        const uint64_t W = st.W;
        auto gpre = [&](uint32_t i) -> uint64_t {
            return st.boff[i / seg] + __ldcg(reinterpret_cast<const unsigned long long *>(&a.item_pre[i]));
        };
        const uint64_t n_chunks = (uint64_t)nwarps * 32;
        const uint64_t my_chunk = warp + (uint64_t)lane * nwarps;
        const uint64_t my_p = (uint64_t)((unsigned __int128)W * my_chunk / n_chunks);
        const uint64_t my_p1 = (uint64_t)((unsigned __int128)W * (my_chunk + 1) / n_chunks);
        uint32_t my_i0 = 0;
        if (my_p < my_p1) {
            uint32_t lo = 0, hi = n_all;            // first item: largest i with gpre(i) <= p
            while (hi - lo > 1) {
                uint32_t mid = lo + (hi - lo) / 2;
                if (gpre(mid) <= my_p) lo = mid; else hi = mid;
            }
            my_i0 = lo;
        }
        // the same search by the whole warp for one pair, 32 probes at a time
        auto item_of = [&](uint64_t p, uint32_t i) {
            for (uint32_t hi = n_all; hi - i > 1;) {
                const uint32_t step = (hi - i + 31) / 32, x = i + lane * step;
                const uint32_t b = __ballot_sync(FULL, x < hi && gpre(x) <= p);
                i += (31 - __clz(b)) * step;                // (lane 0 always holds)
                hi = min(hi, i + step);
            }
            return i;
        };
        const uint32_t wid = threadIdx.x >> 5;
        const bool on_demand = W >= n_chunks * MQ_TAKE_PAIRS;
        const uint32_t n_own = on_demand ? 32 - MQ_TAKE : 32;
        for (uint32_t ch = 0;; ++ch) {
            uint64_t p, p1;
            uint32_t i0;
            if (ch < n_own) {
                p = __shfl_sync(FULL, my_p, ch);
                p1 = __shfl_sync(FULL, my_p1, ch);
                i0 = __shfl_sync(FULL, my_i0, ch);
            } else {
                if (!on_demand) break;
                uint32_t tk = 0;
                if (lane == 0) tk = atomicAdd(&ctl->take[cs], 1u);
                tk = __shfl_sync(FULL, tk, 0);
                if (tk >= MQ_TAKE * nwarps) break;
                const uint64_t chunk = (uint64_t)n_own * nwarps + tk;
                p = (uint64_t)((unsigned __int128)W * chunk / n_chunks);
                p1 = (uint64_t)((unsigned __int128)W * (chunk + 1) / n_chunks);
                i0 = item_of(p, 0);
            }
            while (p < p1) {
                // the window's items, one per lane: arcs, slots and the pairs
                // inside this chunk, left in shared memory for the warp
                uint32_t live;
                {
                    const uint32_t idx = i0 + lane;
                    const uint64_t wend = i0 + 32 < n_all ? gpre(i0 + 32) : W;
                    const uint64_t stop = min(p1, wend);
                    uint64_t pre = wend;
                    uint32_t u = 0, s0 = 0, c = 0;
                    unsigned long long M = 0;
                    const bool hv = idx >= n_items;        // heavy-arc pass item
                    if (idx < n_all) {
                        pre = gpre(idx);
                        u = hv ? ldcg_u32(&blo[idx - n_items]) : ldcg_u32(&qc[idx]);
                        M = __ldcg(&a.item_mask[idx]);
                        s0 = (hv && a.lend) ? a.lend[u] : a.row_ptr[u];
                        c = (uint32_t)popc64(M);
                    }
                    uint64_t end = __shfl_down_sync(FULL, pre, 1);
                    if (lane == 31) end = wend;
                    end = min(end, stop);
                    const uint64_t beg = max(p, pre);
                    const bool has = c != 0 && beg < end;
                    live = __ballot_sync(FULL, has);
                    if (has) {
                        // pair l of the item is (arc l / c, slot l % c)
                        const uint32_t lo = (uint32_t)(beg - pre), hi = (uint32_t)(end - pre);
                        const uint64_t mg = st.mag[c] << 24;
                        const uint32_t jlo = c > 1 ? (uint32_t)__umul64hi((uint64_t)lo, mg) : lo;
                        const uint32_t jhi = c > 1 ? (uint32_t)__umul64hi((uint64_t)(hi - 1), mg) : hi - 1;
                        // heavy-arc items relax weights >= delta, light ones
                        // the rest; bit 8: lower bound, bit 9: upper bound
                        const uint32_t fl = (hv ? 256u : 0u) | (a.defer && !hv && !(M & tails) ? 512u : 0u);
                        st.wa[wid][lane] = make_uint4(u, s0, lo, hi);
                        st.wb[wid][lane] = make_uint4(jlo, jhi, (uint32_t)M, (uint32_t)(M >> 32));
                        st.wc[wid][lane] = c | fl;
                    }
                    __syncwarp();
                    p = stop;
                    i0 += 32;
                }
                // no pair in the window: jump over the items without any.  A
                // band list that one slot of many passes over is full of
                // them, and a warp that walked over a million held up its
                // iteration for 7 to 17 ms.
                if (!live && p < p1) {
                    i0 = item_of(p, i0);
                    continue;
                }
                // The items one after another; the lanes take fixed slots
                // (and, for c <= 16, several arcs per step), so a lane finds
                // its slot and loads the tail's label once per item and then
                // steps over the arcs.
                for (; live; live &= live - 1) {
                    const uint32_t w = __ffs(live) - 1;
                    const uint4 ia = st.wa[wid][w], ib = st.wb[wid][w];
                    const uint32_t ic = st.wc[wid][w], cw = ic & 255u;
                    const uint32_t wlo = ic & 256u ? a.delta : 1u;   // (weight 0: no pair)
                    const uint32_t sw = ia.y, lo = ia.z, hi = ia.w, jhi = ib.y;
                    auto lane_slot = [&](uint32_t tq) {
                        MqLane s{0, 0, INF32, 0, 0};
                        if (tq < cw) {
                            s.q = cw == MQ_SLOTS ? tq : nth_bit64(((unsigned long long)ib.w << 32) | ib.z, tq);
                            s.sh = st.lshift[s.q];
                            s.lab = ldcg_u32(&a.label[(uint64_t)ia.x * MQ_SLOTS + s.q]);
                            s.room = (INF32 >> s.sh) - (s.lab >> s.sh);
                            s.whi = s.lab == INF32 ? 0u : (ic & 512u ? a.delta : INF32);
                        }
                        return s;
                    };
                    if (cw > 32) {
                        // 33..64 slots: each lane takes slots lane and lane + 32
                        const MqLane s0 = lane_slot(lane), s1 = lane_slot(lane + 32);
                        for (uint32_t j0 = ib.x; j0 <= jhi; j0 += MQ_ILP / 2) {
                            uint2 e[MQ_ILP];
#pragma unroll
                            for (int k = 0; k < MQ_ILP; k += 2) {
                                const uint32_t jj = j0 + (uint32_t)(k >> 1), l = jj * cw + lane;
                                uint2 x = make_uint2(0, 0);
                                if (jj <= jhi) x = __ldg(&a.adj[sw + jj]);
                                e[k] = e[k + 1] = x;
                                if (l < lo || l >= hi) e[k].y = 0;
                                if (lane + 32 >= cw || l + 32 < lo || l + 32 >= hi) e[k + 1].y = 0;
                            }
                            mq_relax<true, true>(a, st, t, e, s0, s1, wlo, attempts, improved);
                        }
                    } else {
                        // g lanes per arc (g = c rounded up to a power of two),
                        // 32 / g arcs per step
                        const uint32_t gsh = cw <= 1 ? 0u : 32u - __clz(cw - 1);
                        const uint32_t A = 32u >> gsh;
                        const uint32_t tq = lane & ((1u << gsh) - 1u), aoff = lane >> gsh;
                        const MqLane s0 = lane_slot(tq);
                        for (uint32_t j0 = ib.x; j0 <= jhi; j0 += MQ_ILP * A) {
                            uint2 e[MQ_ILP];
#pragma unroll
                            for (int k = 0; k < MQ_ILP; ++k) {
                                const uint32_t jj = j0 + (uint32_t)k * A + aoff, l = jj * cw + tq;
                                e[k] = make_uint2(0, 0);
                                if (tq < cw && jj <= jhi && l >= lo && l < hi) e[k] = __ldg(&a.adj[sw + jj]);
                            }
                            mq_relax<false, false>(a, st, t, e, s0, s0, wlo, attempts, improved);
                        }
                    }
                }
                __syncwarp();
            }
        }
        if (P) {
            mq_pull_sweep(a, st, P, t.qn, t.qn_count, t.farq, t.far_count, t.tag_next, attempts,
                          improved);
            ++pull_sweeps;
        }
        unsigned long long tm3 = first ? global_ns() : 0;
        seg_flush(st, t, ctl, a.n);
        if (first)
            ctl->stop_req[it & 1] = (a.yield && a.doorbell) ? *(volatile const uint32_t *)a.doorbell : 0u;
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) { reason = 5; break; }
        if (first) {
            unsigned long long tm4 = global_ns();
            ctl->t_part[0] += tm1 - tm0;
            ctl->t_part[1] += tm2 - tm1;
            ctl->t_part[2] += tm3 - tm2;
            ctl->t_part[3] += tm4 - tm3;
            ctl->items_total += n_all;
            ctl->pairs_total += st.W;
        }
        ++it;
        ++iters;
        if (H) bc = (bc + 1) % 3;

        // per-slot decisions (every block computes the same from global
        // state): a slot with near work queued continues its band; an idle
        // one first runs its band's heavy-arc pass (next iteration), then is
        // converged if nothing is parked far, else its far pile is split
        unsigned long long act_next = __ldcg(&ctl->act[it % 3]);
        hp_done &= ~act_next;
        unsigned long long idle = infl & ~act_next, S = 0, conv = 0;
        H = a.defer ? (idle & ~hp_done & ~tails) : 0ull;
        // A pull sweep pays for a slot whose band holds most of the graph.
        const unsigned long long ask = a.pull ? H & band0 & ~wide : 0ull;
        if (ask) {
            const unsigned long long most = mq_wide_bands(a, st, ask, bar_target, reason);
            if (reason) break;
            wide |= ask & (most | late);
            late |= ask & ~most;
        }
        // The sweep visits every vertex however few slots it serves, so
        // drained bands wait (up to MQ_HOLD iterations) for the other slots'
        // and share one sweep.
        const unsigned long long ready = a.pull ? H & band0 & wide : 0ull;
        if (ready && (infl & band0 & (act_next | ~wide)) && held < MQ_HOLD) {
            idle &= ~ready;
            H &= ~ready;
            ++held;
        } else if (ready) {
            held = 0;
        }
        hp_done |= H;
        for (unsigned long long m = idle & ~H; m; m &= m - 1) {
            uint32_t q = __ffsll((long long)m) - 1;
            if (__ldcg(&ctl->far_pending[q]) <= 0) conv |= 1ull << q;
            else S |= 1ull << q;
        }
        infl &= ~conv;
        conv_total |= conv;
        if (!infl) { reason = 1; break; }
        if (a.yield && (uint32_t)popc64(conv_total) >= a.yield) { reason = 2; break; }
        if (a.yield && ldcg_u32(&ctl->stop_req[(it - 1) & 1])) { reason = 3; break; }
        if (iters >= a.max_iters) { reason = 4; break; }
        if (!S) continue;
        // (a launch that left above finds S as it was: the next one decides again)
        hp_done &= ~S;                      // a split opens a new band
        const unsigned long long to_tail = a.pull ? S & band0 & wide : 0ull;
        tails |= to_tail;
        if (a.pull) band0 &= ~to_tail;
        else band0 &= ~S;

        unsigned long long tm5 = first ? global_ns() : 0;
        // Split the far pile for the slots in S.  A barrier first: every
        // block has read the decision inputs before the split appends to
        // them.  Near pushes go to this iteration's queue (slot it % 3).
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) { reason = 5; break; }
        if (threadIdx.x < MQ_SLOTS) {
            uint32_t q = threadIdx.x;
            unsigned long long Tq = st.T[q];
            if ((S >> q) & 1) {
                uint32_t fm = __ldcg(&ctl->fmin[fc][q]);
                unsigned long long base = (fm != INF32 && (unsigned long long)fm > Tq) ? fm : Tq;
                // (a tail has no far side: every parked vertex joins the frontier)
                st.Tnew[q] = (to_tail >> q) & 1 ? 1ull << 40 : base + a.delta;
            } else {
                st.Tnew[q] = Tq;
            }
        }
        seg_reset(st);
        const bool odd2 = it & 1;
        MqTargets u;
        u.qn = odd2 ? a.q1 : a.q0;
        u.qn_count = &ctl->near_count[it % 3];
        u.act = &ctl->act[it % 3];
        u.farq = fc ? a.far0 : a.far1;
        u.far_count = &ctl->far_count[fc ^ 1];
        u.fmin = ctl->fmin[fc ^ 1];
        u.tag_next = a.base_near + it;
        const uint32_t *fs = fc ? a.far1 : a.far0;
        const uint32_t nf = min(ldcg_u32(&ctl->far_count[fc]), a.n);
        for (uint32_t b = warp * 32; b < nf; b += nwarps * 32) {
            uint32_t i = b + lane;
            bool valid = i < nf;
            uint32_t v = valid ? ldcg_u32(&fs[i]) : 0;
            unsigned long long M = valid ? __ldcg(&a.fmask[v]) : 0ull;
            unsigned long long MS = M & S, moved = 0, dropped = 0;
            for (unsigned long long m = MS; m; m &= m - 1) {
                uint32_t q = __ffsll((long long)m) - 1;
                uint64_t d = mq_label(a.label, v, q, st.lshift[q]) >> 32;
                if (d < st.T[q]) {
                    dropped |= 1ull << q;                  // settled while parked
                } else if (d < st.Tnew[q]) {
                    moved |= 1ull << q;
                } else {
                    atomicMin(&st.fmin[q], (uint32_t)d);
                }
            }
            unsigned long long cleared = moved | dropped;
            if (cleared) {
                atomicAnd(&a.fmask[v], ~cleared);
                for (unsigned long long m = cleared; m; m &= m - 1)
                    atomicSub(&st.fpend[__ffsll((long long)m) - 1], 1);
            }
            bool to_near = false;
            if (moved) {
                atomicOr(&a.nmask[v], moved);
                to_near = atomicExch(&a.stamp_near[v], u.tag_next) != u.tag_next;
            }
            unsigned long long act = warp_or64(moved);
            if (lane == 0 && act) atomicOr(&st.act, act);
            bool keep = valid && (M & ~cleared) != 0;
            if (valid && !keep) a.in_far[v] = 0;
            mq_push_near(a, st, u, to_near, v);
            stage_append(keep, v, st.far_buf, &st.far_n, MQ_FAR_STAGE, u.farq, u.far_count, a.n,
                         &ctl->err);
        }
        seg_flush(st, u, ctl, a.n);
        if (!grid_sync(&ctl->bar, &ctl->err, bar_target)) { reason = 5; break; }
        if (first) {
            for (uint32_t q = 0; q < MQ_SLOTS; ++q) {
                if (!((S >> q) & 1)) {
                    uint32_t fm = ctl->fmin[fc][q];
                    if (fm != INF32) atomicMin(&ctl->fmin[fc ^ 1][q], fm);
                }
                ctl->fmin[fc][q] = INF32;
            }
            ctl->far_count[fc] = 0;
        }
        if (threadIdx.x < MQ_SLOTS) st.T[threadIdx.x] = st.Tnew[threadIdx.x];
        __syncthreads();
        fc ^= 1;
        if (first) ctl->t_part[4] += global_ns() - tm5;
    }
    if (!infl && reason == 0) reason = 1;
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
    __syncthreads();
    if (threadIdx.x == 0 && st.miss) atomicOr(&ctl->slot_narrow, st.miss);
    if (first) {
        ctl->it = it;
        ctl->fc = fc;
        ctl->hpass = H & infl;
        ctl->hp_done = hp_done;
        ctl->band0 = band0;
        ctl->wide = wide;
        ctl->late = late;
        ctl->tails = tails;
        ctl->held = held;
        ctl->pull_sweeps += pull_sweeps;
        ctl->blist = bc;
        ctl->converged |= conv_total;
        ctl->iterations = iters;
        ctl->exit_reason = reason;
        for (uint32_t q = 0; q < MQ_SLOTS; ++q) ctl->T[q] = st.T[q];
        if (reason == 4 && infl) atomicOr(&ctl->err, 0u);   // a capped launch resumes later
    }
}

// ---------------------------------------------------------------------------
// admission of one slot: clear its label/pred column, seed it
// ---------------------------------------------------------------------------

__global__ void mq_clear_column_kernel(uint32_t n, uint32_t *label, uint32_t *pred, uint32_t q) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        label[(uint64_t)v * MQ_SLOTS + q] = INF32;
        pred[(uint64_t)v * MQ_SLOTS + q] = INF32;
    }
}

// Clears the label/pred columns of every slot in `mask` with row-wide,
// coalesced stores (one thread per (vertex, slot) element).
__global__ void mq_clear_rows_kernel(uint32_t n, uint32_t *label, uint32_t *pred,
                                     unsigned long long mask) {
    uint64_t total = (uint64_t)n * MQ_SLOTS;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        if ((mask >> (i & (MQ_SLOTS - 1))) & 1ull) {
            label[i] = INF32;
            pred[i] = INF32;
        }
    }
}

// The slots admitted together, one per blockIdx.y: one launch for all (with a
// launch per slot admitting 64 queries took 0.77 ms, now 0.39).
struct MqSeedArgs {
    const int32_t *seeds[MQ_SLOTS];
    uint32_t k[MQ_SLOTS];
    uint32_t q[MQ_SLOTS];
};

__global__ void mq_seed_kernel(uint32_t n, const uint32_t *__restrict__ new_of, uint32_t delta,
                               const __grid_constant__ MqSeedArgs a, const __grid_constant__ MqState m) {
    MqControl *ctl = m.ctl;
    const int32_t *seeds = a.seeds[blockIdx.y];
    const uint32_t k = a.k[blockIdx.y], q = a.q[blockIdx.y];
    uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t it = ctl->it;
    const unsigned long long bit = 1ull << q;
    if (r == 0) {
        uint32_t b = 1;
        while (b < 31 && (1u << b) < k) ++b;
        ctl->lshift[q] = b;
        ctl->T[q] = delta;
        ctl->fmin[0][q] = INF32;
        ctl->fmin[1][q] = INF32;
        ctl->far_pending[q] = 0;
        atomicOr(&ctl->act[it % 3], bit);
        atomicOr(&ctl->band0, bit);
        for (unsigned long long *mask : {&ctl->slot_narrow, &ctl->slot_overflow, &ctl->hp_done, &ctl->hpass,
                                         &ctl->wide, &ctl->late, &ctl->tails})
            atomicAnd(mask, ~bit);
    }
    if (r >= k) return;
    uint32_t s = internal_id(new_of, (uint32_t)seeds[r]);
    m.label[(uint64_t)s * MQ_SLOTS + q] = r;          // distance 0, rank r
    m.pred[(uint64_t)s * MQ_SLOTS + q] = SEED_ARC;
    atomicOr(&m.nmask[s], bit);
    uint32_t tag = m.base_near + it;
    if (atomicExch(&m.stamp_near[s], tag) == tag) return;   // already queued for iteration it
    uint32_t slot = atomicAdd(&ctl->near_count[it % 3], 1u);
    if (slot >= n) {
        atomicOr(&ctl->err, ERR_CAPACITY);
        return;
    }
    ((it & 1) ? m.q[1] : m.q[0])[slot] = s;
}

// ---------------------------------------------------------------------------
// batched pred + bridge scan for a set of converged slots
// ---------------------------------------------------------------------------

struct MqScanArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;
    const uint64_t *__restrict__ heavy_chunks;
    uint32_t n_heavy_chunks;
    const uint32_t *__restrict__ items;   // vertex ranges [items[i], items[i + 1])
    uint32_t n_items;
    uint32_t n;
    const uint32_t *label;
    const uint32_t *lshift;          // rank bits of each slot's labels
    uint32_t *pred;
    uint64_t *const *pairtab;
    const uint32_t *k;
    unsigned long long slots;
    MqControl *ctl;
    const uint32_t *orig_of;         // internal -> caller ids (null: identity)
    const uint32_t *orig_row_ptr;
};

// One slot's view of the row being scanned, held by the lane that serves
// the slot: v's label, and the slot's pair table from the first entry of
// v's cell's row of the upper triangle (pair_slot(cv, cv + 1, k)), so that
// the entry of pair (cv, cu) is tab[cu - cv - 1].
struct ScanSlot {
    uint32_t lv;        // as stored
    uint32_t sh;        // rank bits
    uint64_t *tab;
    uint32_t pmin;      // running minimum of v's pred arc
    uint32_t q;
};

__device__ __forceinline__ ScanSlot mq_row_slot(uint32_t q, uint64_t *tab, uint32_t k, uint32_t sh,
                                                uint32_t lv) {
    ScanSlot r;
    r.lv = lv;
    r.sh = sh;
    r.q = q;
    r.pmin = INF32;
    const uint32_t cv = lv & ((1u << sh) - 1u);
    r.tab = lv == INF32 ? tab : tab + pair_slot(cv, cv + 1, k);
    return r;
}

// Arc `arc` = (v, head, w) for one slot, with lu the slot's label of the head
// and cbase + arc the caller's index of the arc (bridge keys carry it, as in
// the single-query scan).  A tight same-cell arc lowers r.pmin.  Labels are
// compared as stored.
__device__ __forceinline__ void mq_scan_eval(ScanSlot &r, uint32_t arc, uint32_t w, uint32_t lu,
                                             uint32_t cbase, unsigned long long &overflow) {
    if (r.lv == INF32 || lu == INF32) {
        if (r.lv != lu) overflow |= 1ull << r.q;
        return;
    }
    const uint32_t mask = (1u << r.sh) - 1u, cv = r.lv & mask, cu = lu & mask;
    const uint64_t sum = ((uint64_t)w << r.sh) + lu;       // the head's distance + w, its cell
    if (sum == r.lv) {
        r.pmin = min(r.pmin, arc);
    } else if (cv < cu) {
        const uint64_t b = (r.lv >> r.sh) + (sum >> r.sh);
        if (b >= INF32) {
            overflow |= 1ull << r.q;
            return;
        }
        const uint64_t key = (b << 32) | (uint32_t)(cbase + arc);
        uint64_t *slot = r.tab + (cu - cv - 1);
        // a cached read may be stale, i.e. larger: at worst one atomic more
        if (key < __ldg(reinterpret_cast<const unsigned long long *>(slot)))
            atomicMin(reinterpret_cast<unsigned long long *>(slot), (unsigned long long)key);
    }
}

__device__ __forceinline__ void mq_store_pred(const MqScanArgs &a, uint32_t v, const ScanSlot &r,
                                              bool whole_row) {
    if (r.pmin == INF32) return;
    uint32_t *pp = &a.pred[(uint64_t)v * MQ_SLOTS + r.q];
    if (whole_row) *pp = r.pmin;
    else atomicMin(pp, r.pmin);
}

// Label runs in flight per warp in the slot-pair mode.  The scan is bound by
// the evaluation of (arc, slot) pairs and the probes of the pair tables (R-MAT
// 22 x 64 queries: 17.1 ms; 7.6 with the label runs alone): labels compared
// as stored and cached probes took it down from 22.4.
constexpr int SCAN_ARCS = 4;

// The slots a lane serves for the whole launch, with their pair tables and
// sizes loaded once.
struct LaneSlots {
    uint32_t q0, k0, k1;
    uint32_t sh0, sh1;      // rank bits of the slots' labels
    bool h0, h1;
    uint64_t *t0, *t1;
};

// A piece of one vertex's arcs for every slot of the launch.  Each lane keeps
// its slots' row state in registers and stores v's pred once per slot
// (atomically when the row is split into chunks over several warps).
// Over 32 slots: lane l takes slots 2l and 2l + 1 (one 8-byte load of the
// pair's labels per arc), and every lane walks every arc.
// Otherwise lanes are grouped as in the SSSP kernel: a group of g lanes
// takes one arc, lane t of the group the t-th slot; the groups' minima meet
// by shuffles.
__device__ __forceinline__ void mq_scan_row(const MqScanArgs &a, const LaneSlots &ls, uint32_t v,
                                            uint32_t rs, RowPiece p, bool whole_row,
                                            uint32_t cnt, uint32_t gsh,
                                            unsigned long long &overflow) {
    const uint32_t lane = lane_id();
    const uint32_t cbase = caller_arc_base(a.orig_of, a.orig_row_ptr, v, rs);
    const uint32_t *lrow = &a.label[(uint64_t)v * MQ_SLOTS];
    if (cnt > 32) {
        const uint2 lv = __ldg(reinterpret_cast<const uint2 *>(&lrow[ls.q0]));
        ScanSlot r0 = mq_row_slot(ls.q0, ls.t0, ls.k0, ls.sh0, lv.x);
        ScanSlot r1 = mq_row_slot(ls.q0 + 1, ls.t1, ls.k1, ls.sh1, lv.y);
        // the arc records 32 at a time, one per lane, streamed
        const uint32_t end = p.first + p.count;
        for (uint32_t w0 = p.first, got; w0 != end; w0 += got) {     // (end + 31 may wrap)
            got = min(32u, end - w0);
            uint2 mine = make_uint2(0, 0);
            if (lane < got) mine = __ldcs(&a.adj[w0 + lane]);
            for (uint32_t i = 0; i < got; i += SCAN_ARCS) {
                uint2 lu[SCAN_ARCS];
#pragma unroll
                for (int k = 0; k < SCAN_ARCS; ++k) {
                    const uint32_t head = __shfl_sync(FULL, mine.x, i + k);
                    lu[k] = make_uint2(INF32, INF32);
                    if (i + k < got)
                        lu[k] = __ldg(reinterpret_cast<const uint2 *>(
                            &a.label[(uint64_t)head * MQ_SLOTS + ls.q0]));
                }
#pragma unroll
                for (int k = 0; k < SCAN_ARCS; ++k) {
                    const uint32_t w = __shfl_sync(FULL, mine.y, i + k);
                    if (i + k >= got) break;
                    if (ls.h0) mq_scan_eval(r0, w0 + i + k, w, lu[k].x, cbase, overflow);
                    if (ls.h1) mq_scan_eval(r1, w0 + i + k, w, lu[k].y, cbase, overflow);
                }
            }
        }
        if (ls.h0) mq_store_pred(a, v, r0, whole_row);
        if (ls.h1) mq_store_pred(a, v, r1, whole_row);
        return;
    }
    const uint32_t g = 1u << gsh, apr = 32 >> gsh, grp = lane >> gsh;
    const bool has_slot = ls.h0;
    ScanSlot r = mq_row_slot(ls.q0, ls.t0, ls.k0, ls.sh0, has_slot ? __ldg(&lrow[ls.q0]) : INF32);
    for (; p.count; skip_arcs(p, apr * 4)) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t j = k * apr + grp, arc = p.first + j;
            if (has_slot && j < p.count) {
                uint2 e = __ldg(&a.adj[arc]);
                const uint32_t lu = __ldg(&a.label[(uint64_t)e.x * MQ_SLOTS + ls.q0]);
                mq_scan_eval(r, arc, e.y, lu, cbase, overflow);
            }
        }
    }
    for (uint32_t off = g; off < 32; off <<= 1)
        r.pmin = min(r.pmin, __shfl_xor_sync(FULL, r.pmin, off));
    if (grp == 0 && has_slot) mq_store_pred(a, v, r, whole_row);
}

__global__ void __launch_bounds__(256, 5) mq_scan_kernel(MqScanArgs a) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t cnt = (uint32_t)popc64(a.slots);
    const uint32_t gsh = cnt > 16 ? 5 : cnt > 8 ? 4 : cnt > 4 ? 3 : cnt > 2 ? 2 : cnt > 1 ? 1 : 0;
    LaneSlots ls;
    if (cnt > 32) {
        ls.q0 = 2 * lane;
        ls.h0 = (a.slots >> ls.q0) & 1;
        ls.h1 = (a.slots >> (ls.q0 + 1)) & 1;
    } else {
        const uint32_t tl = lane & ((1u << gsh) - 1);
        ls.h0 = tl < cnt;
        ls.h1 = false;
        ls.q0 = ls.h0 ? nth_bit64(a.slots, tl) : 0;
    }
    ls.t0 = ls.h0 ? a.pairtab[ls.q0] : nullptr;
    ls.k0 = ls.h0 ? a.k[ls.q0] : 0;
    ls.t1 = ls.h1 ? a.pairtab[ls.q0 + 1] : nullptr;
    ls.k1 = ls.h1 ? a.k[ls.q0 + 1] : 0;
    ls.sh0 = ls.h0 ? a.lshift[ls.q0] : 1;
    ls.sh1 = ls.h1 ? a.lshift[ls.q0 + 1] : 1;
    const uint32_t n_work = a.n_heavy_chunks + a.n_items;
    unsigned long long overflow = 0;
    for (uint32_t wi = warp; wi < n_work; wi += nwarps) {
        if (wi < a.n_heavy_chunks) {
            uint64_t item = a.heavy_chunks[wi];
            uint32_t v = (uint32_t)(item >> 32), c = (uint32_t)item;
            uint32_t rs = a.row_ptr[v];
            mq_scan_row(a, ls, v, rs, row_piece(rs, a.row_ptr[v + 1], c * CHUNK, CHUNK), false, cnt, gsh,
                        overflow);
        } else {
            const uint32_t v1 = __ldg(&a.items[wi - a.n_heavy_chunks + 1]);
            for (uint32_t v0 = __ldg(&a.items[wi - a.n_heavy_chunks]); v0 < v1; v0 += 32) {
                const uint32_t vl = v0 + lane;
                const uint32_t rs = vl < v1 ? a.row_ptr[vl] : 0;
                const uint32_t re = vl < v1 ? a.row_ptr[vl + 1] : 0;
                for (uint32_t l = 0; l < 32 && v0 + l < v1; ++l) {
                    const uint32_t s = __shfl_sync(FULL, rs, l), e = __shfl_sync(FULL, re, l);
                    // hubs are covered by the chunk list; no arcs, nothing to scan
                    if (e - s >= HEAVY_DEG || e == s) continue;
                    mq_scan_row(a, ls, v0 + l, s, RowPiece{s, e - s}, true, cnt, gsh, overflow);
                }
            }
        }
    }
    overflow = warp_or64(overflow);
    if (lane == 0 && overflow) atomicOr(&a.ctl->slot_overflow, overflow);
}

// ---------------------------------------------------------------------------
// the scan of slots that return the tree alone
// ---------------------------------------------------------------------------
//
// As in the single-query tree-only scan: mq_tree_scan_kernel reads the light
// part of the rows, for the predecessors of the (vertex, slot) pairs nearer
// than delta and for every bridge below delta, and whole rows only for the
// predecessors of the vertices that are farther in some slot; the batched
// tails form each slot's MST of those pairs; mq_rest_scan_kernel then reads
// the rows of the (vertex, slot) pairs outside the cells of the slot's hub
// component (the one with most arcs), and the MST of all pairs found is the
// slot's MST of G'_1.  A predecessor is an index in the rows split by weight
// for a pair nearer than delta, in the caller's order for another.
//
// The full scan evaluates every (arc, slot) pair and is bound by that; here a
// light arc is a few 32-bit operations and most bridges fail b < delta before
// the table is probed.  R-MAT 22, 64 queries: scan 17.1 -> 4.3 ms, tails with
// the rest scan and the second MST 0.5 -> 1.3 ms, batch 44.0 -> 32.2 ms; R-MAT
// 20, serving 90: 28-36 -> 25-34 ms.  It pays from about eight slots on, a
// little later on small graphs: 8 slots R-MAT 20 6.1 against 5.8 ms, R-MAT 22
// 19.2 against 20.3; 12 slots 6.7 against 7.0 and 22.5 against 25.4 (the line,
// MQ_TREE_SLOTS, lies between).  24 and 64 slots, weights to 20 and up to 1000:
// 1.00 to 1.45 times as fast.  Slots whose first band covered little are left
// to the full scan: each would have nearly every whole row read (scan 4.3 ->
// 9.5 ms with one to five of them, 7.5 with the full scan for these).  Exact as
// in the single-query path: two rank bits or more rule out that a bridge
// overflows.

struct MqTreeArgs {
    const uint32_t *__restrict__ row_ptr;
    const uint2 *__restrict__ adj;
    const uint2 *__restrict__ adj_w;
    const uint32_t *__restrict__ lend;
    const uint64_t *__restrict__ heavy_chunks;
    uint32_t n_heavy_chunks;
    const uint32_t *__restrict__ items;
    uint32_t n_items;
    uint32_t delta;
    const uint32_t *label;
    const uint32_t *lshift;
    uint32_t *pred;
    uint64_t *const *pairtab;
    const uint32_t *k;
    unsigned long long slots;
    const uint32_t *orig_of, *orig_row_ptr;
    const TailSlot *tails;           // rest scan: the retiring slots,
    const TailOut *out;              // their hub components
    const uint32_t *comp;            // and the component of every cell
    uint32_t r;
};

// Proposes bridge b over arc x -> y for a table entry (x in the cell of smaller
// rank); the key's arc is searched only if the entry goes down.
__device__ __forceinline__ void mq_propose(const MqTreeArgs &a, uint64_t *entry, uint64_t b,
                                           uint32_t x, uint32_t y) {
    auto *slot = reinterpret_cast<unsigned long long *>(entry);
    if (b > __ldg(slot) >> 32) return;
    if (b > atomicMin(slot, (b << 32) | INF32) >> 32) return;
    const uint32_t rs = a.row_ptr[x], want = caller_id(a.orig_of, y);
    uint32_t lo = rs, hi = a.row_ptr[x + 1];
    while (hi - lo > 1) {                // largest arc whose head is at or before y
        const uint32_t mid = lo + (hi - lo) / 2;
        if (caller_id(a.orig_of, a.adj[mid].x) <= want) lo = mid;
        else hi = mid;
    }
    atomicMin(slot, (b << 32) | (uint32_t)(caller_arc_base(a.orig_of, a.orig_row_ptr, x, rs) + lo));
}

// A slot served by a lane for the whole launch.
struct TreeSlot {
    uint32_t q, sh, k;
    uint64_t *tab;
    bool on;
};

__device__ __forceinline__ TreeSlot tree_slot(const MqTreeArgs &a, uint32_t q) {
    TreeSlot t{q, 1u, 0u, nullptr, ((a.slots >> q) & 1ull) != 0};
    if (t.on) {
        t.sh = a.lshift[q];
        t.k = a.k[q];
        t.tab = a.pairtab[q];
    }
    return t;
}

// Light arc `arc` = (v, y, w) for a slot with v's label lv below the near
// limit: `limit` is that limit, or 0 for a slot that does not look.
__device__ __forceinline__ void tree_light(const MqTreeArgs &a, const TreeSlot &t, uint32_t lv,
                                           uint32_t limit, uint32_t v, uint32_t y, uint32_t w,
                                           uint32_t lu, uint32_t arc, uint32_t &pmin) {
    if (lu >= limit) return;
    const uint32_t sum = lu + (w << t.sh);           // (both below 2^31)
    if (sum == lv) pmin = min(pmin, arc);
    const uint32_t b = (lv >> t.sh) + (sum >> t.sh);
    if (b >= a.delta) return;
    const uint32_t mask = (1u << t.sh) - 1u, cv = lv & mask, cu = lu & mask;
    if (cv < cu) mq_propose(a, t.tab + pair_slot(cv, cu, t.k), b, v, y);
}

// Arcs [s0, s1) of `arcs`, every lane walking every arc: fn(arc, head, w,
// labels of the head for the lane's two slots).
template <class F>
__device__ __forceinline__ void tree_arcs(const MqTreeArgs &a, const uint2 *__restrict__ arcs,
                                          uint32_t s0, uint32_t s1, bool look, F fn) {
    const uint32_t lane = lane_id();
    for (uint32_t w0 = s0; w0 < s1; w0 += 32) {      // (cannot wrap: MQ_TREE_MAX_ARCS)
        uint2 mine = make_uint2(0, 0);
        if (w0 + lane < s1) mine = __ldcs(&arcs[w0 + lane]);
        const uint32_t got = min(32u, s1 - w0);
        for (uint32_t i = 0; i < got; i += SCAN_ARCS) {
            uint2 lu[SCAN_ARCS];
#pragma unroll
            for (int j = 0; j < SCAN_ARCS; ++j) {
                const uint32_t head = __shfl_sync(FULL, mine.x, i + j);
                lu[j] = make_uint2(INF32, INF32);
                if (look && i + j < got)
                    lu[j] = __ldg(reinterpret_cast<const uint2 *>(
                        &a.label[(uint64_t)head * MQ_SLOTS + 2 * lane]));
            }
#pragma unroll
            for (int j = 0; j < SCAN_ARCS; ++j) {
                const uint32_t y = __shfl_sync(FULL, mine.x, i + j), w = __shfl_sync(FULL, mine.y, i + j);
                if (i + j < got) fn(w0 + i + j, y, w, lu[j]);
            }
        }
    }
}

// Calls fn(v, first arc, row end, hub piece?, v's labels) for every row that is
// not empty and for every CHUNK-arc piece of a hub row; the labels of
// a row are fetched a row ahead.
template <class F>
__device__ __forceinline__ void tree_rows(const MqTreeArgs &a, F fn) {
    const uint32_t lane = lane_id();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t n_work = a.n_heavy_chunks + a.n_items;
    auto labels = [&](uint32_t v) {
        return __ldg(reinterpret_cast<const uint2 *>(&a.label[(uint64_t)v * MQ_SLOTS + 2 * lane]));
    };
    for (uint32_t wi = warp; wi < n_work; wi += nwarps) {
        if (wi < a.n_heavy_chunks) {
            const uint64_t item = a.heavy_chunks[wi];
            const uint32_t v = (uint32_t)(item >> 32);
            fn(v, a.row_ptr[v] + (uint32_t)item * CHUNK, a.row_ptr[v + 1], true, labels(v));
            continue;
        }
        const uint32_t v1 = __ldg(&a.items[wi - a.n_heavy_chunks + 1]);
        for (uint32_t v0 = __ldg(&a.items[wi - a.n_heavy_chunks]); v0 < v1; v0 += 32) {
            const uint32_t vl = v0 + lane;
            const uint32_t rs = vl < v1 ? a.row_ptr[vl] : 0;
            const uint32_t re = vl < v1 ? a.row_ptr[vl + 1] : 0;
            uint32_t rows = __ballot_sync(FULL, re - rs < HEAVY_DEG && re != rs);
            uint2 next = rows ? labels(v0 + __ffs(rows) - 1) : make_uint2(0, 0);
            while (rows) {
                const uint32_t l = __ffs(rows) - 1;
                const uint2 lv = next;
                rows &= rows - 1;
                if (rows) next = labels(v0 + __ffs(rows) - 1);
                fn(v0 + l, __shfl_sync(FULL, rs, l), __shfl_sync(FULL, re, l), false, lv);
            }
        }
    }
}

__global__ void __launch_bounds__(256, 5) mq_tree_scan_kernel(const __grid_constant__ MqTreeArgs a) {
    const TreeSlot t0 = tree_slot(a, 2 * lane_id()), t1 = tree_slot(a, 2 * lane_id() + 1);
    const uint32_t n0 = t0.on ? a.delta << t0.sh : 0u, n1 = t1.on ? a.delta << t1.sh : 0u;
    tree_rows(a, [&](uint32_t v, uint32_t s, uint32_t re, bool hub, uint2 lv) {
        const uint32_t l0 = lv.x < n0 ? n0 : 0u, l1 = lv.y < n1 ? n1 : 0u;
        const bool f0 = t0.on && lv.x >= n0 && lv.x != INF32, f1 = t1.on && lv.y >= n1 && lv.y != INF32;
        uint32_t p0 = INF32, p1 = INF32;
        if (__any_sync(FULL, l0 | l1)) {
            tree_arcs(a, a.adj_w, s, piece_end(s, a.lend[v], CHUNK), l0 | l1, [&](uint32_t arc, uint32_t y, uint32_t w, uint2 lu) {
                tree_light(a, t0, lv.x, l0, v, y, w, lu.x, arc, p0);
                tree_light(a, t1, lv.y, l1, v, y, w, lu.y, arc, p1);
            });
        }
        if (__any_sync(FULL, f0 || f1)) {
            tree_arcs(a, a.adj, s, piece_end(s, re, CHUNK), f0 || f1, [&](uint32_t arc, uint32_t, uint32_t w, uint2 lu) {
                if (f0 && w <= lv.x >> t0.sh && lv.x - (w << t0.sh) == lu.x) p0 = min(p0, arc);
                if (f1 && w <= lv.y >> t1.sh && lv.y - (w << t1.sh) == lu.y) p1 = min(p1, arc);
            });
        }
        uint32_t *pp = &a.pred[(uint64_t)v * MQ_SLOTS + t0.q];
        if (p0 != INF32) { if (hub) atomicMin(pp, p0); else *pp = p0; }
        if (p1 != INF32) { if (hub) atomicMin(pp + 1, p1); else pp[1] = p1; }
    });
}

__global__ void __launch_bounds__(256, 5) mq_rest_scan_kernel(const __grid_constant__ MqTreeArgs a) {
    __shared__ uint32_t s_hub[MQ_SLOTS], s_comp0[MQ_SLOTS];
    if (threadIdx.x < a.r) {
        const TailSlot &sl = a.tails[threadIdx.x];
        s_hub[sl.q] = a.out[threadIdx.x].hub;
        s_comp0[sl.q] = sl.comp0;
    }
    __syncthreads();
    const TreeSlot t0 = tree_slot(a, 2 * lane_id()), t1 = tree_slot(a, 2 * lane_id() + 1);
    auto comp = [&](const TreeSlot &t, uint32_t l) {
        return __ldg(&a.comp[s_comp0[t.q] + (l & ((1u << t.sh) - 1u))]);
    };
    tree_rows(a, [&](uint32_t v, uint32_t s, uint32_t re, bool hub, uint2 lv) {
        uint32_t c0 = 0, c1 = 0;
        bool o0 = t0.on && lv.x != INF32, o1 = t1.on && lv.y != INF32;
        if (o0) o0 = (c0 = comp(t0, lv.x)) != s_hub[t0.q];
        if (o1) o1 = (c1 = comp(t1, lv.y)) != s_hub[t1.q];
        if (!__any_sync(FULL, o0 || o1)) return;
        auto arc_of = [&](const TreeSlot &t, uint32_t l, uint32_t c, uint32_t y, uint32_t w, uint32_t lu) {
            if (lu == INF32 || comp(t, lu) == c) return;
            const uint32_t mask = (1u << t.sh) - 1u, cv = l & mask, cu = lu & mask;
            const uint64_t b = (uint64_t)(l >> t.sh) + w + (lu >> t.sh);
            // (in the other cell's row the arc may not be read)
            if (cv < cu) mq_propose(a, t.tab + pair_slot(cv, cu, t.k), b, v, y);
            else mq_propose(a, t.tab + pair_slot(cu, cv, t.k), b, y, v);
        };
        tree_arcs(a, a.adj, s, piece_end(s, re, CHUNK), o0 || o1, [&](uint32_t, uint32_t y, uint32_t w, uint2 lu) {
            if (o0) arc_of(t0, lv.x, c0, y, w, lu.x);
            if (o1) arc_of(t1, lv.y, c1, y, w, lu.y);
        });
    });
}

// Takes the slots' predecessors and pairs back to none, before the full scan.
__global__ void mq_forget_kernel(uint32_t n, const uint32_t *label, const uint32_t *lshift, uint32_t *pred,
                                 unsigned long long mask) {
    const uint64_t total = (uint64_t)n * MQ_SLOTS;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t q = (uint32_t)i & (MQ_SLOTS - 1);
        if ((mask >> q) & 1ull) pred[i] = label[i] >> lshift[q] ? INF32 : SEED_ARC;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

template <class T>
static cudaError_t mq_dalloc(T *&p, uint64_t count) {
    if (count == 0) count = 1;
    return cudaMalloc((void **)&p, count * sizeof(T));
}

cudaError_t mq_alloc(const DevGraph &g, MqState &m, cudaStream_t s) {
    uint32_t n = g.n;
    m.n = n;
    cudaError_t e;
#define MA(ptr, cnt) if ((e = mq_dalloc(ptr, cnt)) != cudaSuccess) return e
    MA(m.label, (uint64_t)n * MQ_SLOTS);      // 32-bit labels
    MA(m.pred, (uint64_t)n * MQ_SLOTS);
    MA(m.nmask, n);
    MA(m.fmask, n);
    MA(m.stamp_near, n);
    MA(m.in_far, n);
    for (int i = 0; i < 2; ++i) {
        MA(m.q[i], n);
        MA(m.far[i], n);
    }
    MA(m.item_mask, 2 * (uint64_t)n);
    MA(m.item_pre, 2 * (uint64_t)n);
    MA(m.bmask, n);
    for (int i = 0; i < 3; ++i) MA(m.bl[i], n);
    MA(m.bsum, MQ_MAX_BLOCKS);
    MA(m.ctl, 1);
    MA(m.d_pairtab, MQ_SLOTS);
    MA(m.d_k, MQ_SLOTS);
#undef MA
    if ((e = mq_reset(m, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(m.d_pairtab, 0, MQ_SLOTS * sizeof(uint64_t *), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(m.d_k, 0, MQ_SLOTS * 4, s)) != cudaSuccess) return e;
    m.base_near = 1;
    return cudaSuccess;
}

cudaError_t mq_reset(MqState &m, cudaStream_t s) {
    const size_t n = m.n;
    cudaError_t e = cudaMemsetAsync(m.nmask, 0, n * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.fmask, 0, n * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.bmask, 0, n * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.stamp_near, 0, n * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.in_far, 0, n * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(m.ctl, 0, sizeof(MqControl), s);
    return e;
}

void mq_free(MqState &m) {
    void *bufs[] = {m.label, m.pred, m.nmask, m.fmask, m.stamp_near, m.in_far, m.q[0], m.q[1],
                    m.item_mask, m.item_pre, m.bsum, m.far[0], m.far[1], m.ctl, m.d_pairtab,
                    m.d_k, m.bmask, m.bl[0], m.bl[1], m.bl[2]};
    for (void *p : bufs)
        if (p) cudaFree(p);
    for (int q = 0; q < MQ_SLOTS; ++q) {
        if (m.pairtab[q]) cudaFree(m.pairtab[q]);
        if (m.seeds[q]) cudaFree(m.seeds[q]);
    }
    m = MqState();
}

int mq_occupancy(int threads) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, mq_sssp_kernel, threads, 0) != cudaSuccess)
        return 0;
    return nb;
}

cudaError_t mq_launch_clear(const DevGraph &g, MqState &m, unsigned long long mask,
                            cudaStream_t s) {
    if (!mask) return cudaSuccess;
    if (__builtin_popcountll(mask) >= 8) {
        mq_clear_rows_kernel<<<current_sm_count() * 16, 256, 0, s>>>(g.n, m.label, m.pred, mask);
    } else {
        unsigned grid = (unsigned)std::min<uint64_t>((g.n + 255) / 256, (uint64_t)current_sm_count() * 16);
        for (unsigned long long mm = mask; mm; mm &= mm - 1)
            mq_clear_column_kernel<<<grid, 256, 0, s>>>(g.n, m.label, m.pred,
                                                        (uint32_t)__builtin_ctzll(mm));
    }
    return cudaGetLastError();
}

cudaError_t mq_launch_seed(const DevGraph &g, MqState &m, unsigned long long slots, const uint32_t *ks,
                           uint32_t delta, cudaStream_t s) {
    MqSeedArgs a{};
    uint32_t r = 0, most = 1;
    for (unsigned long long mm = slots; mm; mm &= mm - 1, ++r) {
        const int q = __builtin_ctzll(mm);
        a.seeds[r] = m.seeds[q];
        a.k[r] = ks[q];
        a.q[r] = (uint32_t)q;
        most = std::max(most, ks[q]);
    }
    if (!r) return cudaSuccess;
    mq_seed_kernel<<<dim3((most + 255) / 256, r), 256, 0, s>>>(g.n, g.new_of, delta, a, m);
    return cudaGetLastError();
}

cudaError_t mq_launch_sssp(const DevGraph &g, MqState &m, int blocks, uint32_t delta, uint32_t pull,
                           uint32_t max_iters, uint32_t yield, const uint32_t *doorbell,
                           cudaStream_t s) {
    MqArgs a;
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.n = g.n;
    a.label = m.label;
    a.nmask = m.nmask;
    a.fmask = m.fmask;
    a.stamp_near = m.stamp_near;
    a.in_far = m.in_far;
    a.q0 = m.q[0];
    a.q1 = m.q[1];
    a.item_mask = m.item_mask;
    a.item_pre = m.item_pre;
    a.bsum = m.bsum;
    a.far0 = m.far[0];
    a.far1 = m.far[1];
    a.bmask = m.bmask;
    a.bl0 = m.bl[0];
    a.bl1 = m.bl[1];
    a.bl2 = m.bl[2];
    a.defer = delta <= g.max_w ? 1u : 0u;
    a.lend = active_lend(g, delta);
    if (a.lend) a.adj = g.adj_w;        // rows partitioned by weight class
    a.pull = a.defer ? pull : 0u;
    a.heavy_chunks = g.heavy_chunks;
    a.n_heavy_chunks = g.n_heavy_chunks;
    a.ctl = m.ctl;
    a.doorbell = doorbell;
    a.delta = delta;
    a.base_near = m.base_near;
    a.max_iters = max_iters;
    a.yield = yield;
    cudaError_t e = cudaMemsetAsync(&m.ctl->bar, 0, sizeof(GridBarrier), s);
    if (e != cudaSuccess) return e;
    if (blocks > MQ_MAX_BLOCKS) blocks = MQ_MAX_BLOCKS;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel((const void *)mq_sssp_kernel, dim3(blocks), dim3(256), args,
                                       0, s);
}

cudaError_t mq_launch_scan(const DevGraph &g, MqState &m, unsigned long long slots,
                           cudaStream_t s) {
    if (!slots) return cudaSuccess;
    MqScanArgs a;
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.heavy_chunks = g.heavy_chunks;
    a.n_heavy_chunks = g.n_heavy_chunks;
    a.items = g.scan_items();
    a.n_items = g.n_scan_items();
    a.n = g.n;
    a.label = m.label;
    a.lshift = m.ctl->lshift;
    a.pred = m.pred;
    a.pairtab = m.d_pairtab;
    a.k = m.d_k;
    a.slots = slots;
    a.ctl = m.ctl;
    a.orig_of = g.orig_of;
    a.orig_row_ptr = g.orig_row_ptr;
    uint64_t work = (uint64_t)g.n_heavy_chunks + g.n_scan_items();
    uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((work + 7) / 8, (uint64_t)current_sm_count() * 32));
    mq_scan_kernel<<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

static MqTreeArgs mq_tree_args(const DevGraph &g, MqState &m, unsigned long long slots, uint32_t delta) {
    MqTreeArgs a{};
    a.row_ptr = g.row_ptr;
    a.adj = g.adj;
    a.adj_w = g.adj_w;
    a.lend = active_lend(g, delta);
    a.heavy_chunks = g.heavy_chunks;
    a.n_heavy_chunks = g.n_heavy_chunks;
    a.items = g.scan_items();
    a.n_items = g.n_scan_items();
    a.delta = delta;
    a.label = m.label;
    a.lshift = m.ctl->lshift;
    a.pred = m.pred;
    a.pairtab = m.d_pairtab;
    a.k = m.d_k;
    a.slots = slots;
    a.orig_of = g.orig_of;
    a.orig_row_ptr = g.orig_row_ptr;
    return a;
}

static unsigned mq_tree_blocks(const DevGraph &g) {
    const uint64_t work = (uint64_t)g.n_heavy_chunks + g.n_scan_items();
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((work + 7) / 8, (uint64_t)current_sm_count() * 32));
}

bool mq_tree_scan_applies(const DevGraph &g, uint32_t k, uint32_t delta) {
    uint32_t b = 1;
    while (b < 31 && (1u << b) < k) ++b;
    return b >= 2 && g.max_w < 0x80000000u && active_lend(g, delta) && delta < 1ull << (31 - b) &&
           g.m <= MQ_TREE_MAX_ARCS;
}

cudaError_t mq_launch_tree_scan(const DevGraph &g, MqState &m, unsigned long long slots, uint32_t delta,
                                cudaStream_t s) {
    const MqTreeArgs a = mq_tree_args(g, m, slots, delta);
    mq_tree_scan_kernel<<<mq_tree_blocks(g), 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t mq_launch_rest_scan(const DevGraph &g, MqState &m, unsigned long long slots, uint32_t delta,
                                const TailSlot *tails, const TailOut *out, const uint32_t *comp, uint32_t r,
                                cudaStream_t s) {
    MqTreeArgs a = mq_tree_args(g, m, slots, delta);
    a.tails = tails;
    a.out = out;
    a.comp = comp;
    a.r = r;
    mq_rest_scan_kernel<<<mq_tree_blocks(g), 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t mq_launch_forget(const DevGraph &g, MqState &m, unsigned long long slots, const uint32_t *ks,
                             cudaStream_t s) {
    mq_forget_kernel<<<current_sm_count() * 8, 256, 0, s>>>(g.n, m.label, m.ctl->lshift, m.pred, slots);
    cudaError_t e = cudaGetLastError();
    for (unsigned long long mm = slots; mm && e == cudaSuccess; mm &= mm - 1) {
        const int q = __builtin_ctzll(mm);
        const uint64_t n_slots = (uint64_t)ks[q] * (ks[q] - 1) / 2;
        if (n_slots) e = cudaMemsetAsync(m.pairtab[q], 0xFF, n_slots * 8, s);
    }
    return e;
}

}  // namespace stn
