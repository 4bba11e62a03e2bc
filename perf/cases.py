"""Performance cases of the Steiner-tree library: what its users call, over
the range of sizes they call it with.

A case names an entry point (``kind``), a seeded synthetic graph and a seed
count.  Graphs are the two families of the evaluation workloads: scale-free
R-MAT graphs (a, b, c = 0.57, 0.19, 0.19) and 4-connected grids, with integer
weights uniform in [1, wmax] and seeds uniform over the component of the
largest hub (every vertex of a grid).  ``n`` need not be a power of two: the
R-MAT ids are scaled down onto [0, n).

kinds
  query    steiner_query: host seeds in, tree edges and total out
  detail   steiner_query_detail with the distance graph G'_1
  voronoi  steiner_voronoi into device tensors (cell, dist, pred)
  noalloc  steiner_voronoi_noalloc on caller-owned device arrays
  batch    steiner_query_batch of many seed sets of uneven size
  serve    steiner_submit of a burst of queries, steiner_poll until all are in

``tuned`` = 1 sets what the autotuner settles on for such graphs (a sixteenth
of the default band width on R-MAT, 32 local rounds on grids); 0 leaves a
handle's defaults.  The graph, its handle, the output buffers and the running
server are what a program keeps; one pass is one call.  All results are exact
integers.
"""
import math
import time

import numpy as np
import torch

from paper_2205_14503_gb300 import steiner as st

ABC = (0.57, 0.19, 0.19)


def listed():
    return [
        # the smallest call: a few thousand vertices, all latency and launches
        dict(name="query_rmat12_k12", kind="query", graph="rmat", n=4096, degree=8, wmax=100, k=12, tuned=0),
        # the plain single-query workload
        dict(name="query_rmat16_k16", kind="query", graph="rmat", n=65536, degree=16, wmax=100, k=16, tuned=0),
        # an ordinary graph of a ragged size at a handle's defaults
        dict(name="query_rmat_ragged_k101", kind="query", graph="rmat", n=1000003, degree=16, wmax=1000, k=101, tuned=0),
        # the largest: 10,000 seeds on a billion arcs, labels beyond the L2 cache, tuned
        dict(name="query_rmat26_k10000", kind="query", graph="rmat", n=1 << 26, degree=8, wmax=1000, k=10000, tuned=1),
        # a mid-size ragged grid (high diameter) at a handle's defaults
        dict(name="query_grid1021x733_k37", kind="query", graph="grid", width=1021, height=733, wmax=1000, k=37, tuned=0),
        # the plain high-diameter workload, tuned
        dict(name="query_grid4096_k256", kind="query", graph="grid", width=4096, height=4096, wmax=1000, k=256, tuned=1),
        # many seeds, with the whole distance graph returned
        dict(name="detail_rmat20_k1000", kind="detail", graph="rmat", n=1 << 20, degree=16, wmax=1000, k=1000, tuned=0),
        # cells, distances and predecessors on the device, wide weights
        dict(name="voronoi_rmat22_k64_w100000", kind="voronoi", graph="rmat", n=1 << 22, degree=16, wmax=100000, k=64, tuned=1),
        # a caller that owns all device memory
        dict(name="noalloc_rmat_n200003_k300", kind="noalloc", graph="rmat", n=200003, degree=16, wmax=1000, k=300, tuned=0),
        dict(name="noalloc_grid499x401_k25", kind="noalloc", graph="grid", width=499, height=401, wmax=1000, k=25, tuned=0),
        # the batched workload: 64 queries of 3 to 1000 seeds, one resident graph
        dict(name="batch_rmat22_q64", kind="batch", graph="rmat", n=1 << 22, degree=16, wmax=1000, queries=64, klo=3, khi=1000, tuned=1),
        # a burst larger than the engine's slots through the serving calls
        dict(name="serve_rmat20_q90", kind="serve", graph="rmat", n=1 << 20, degree=16, wmax=1000, queries=90, klo=3, khi=3000, tuned=1),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["query"] * 4 + ["detail", "voronoi", "voronoi", "noalloc", "noalloc", "batch", "batch", "serve"])
    many = kind in ("batch", "serve")
    graph = "grid" if rng.random() < 1 / 3 else "rmat"
    top = {"query": 24, "voronoi": 24, "detail": 22, "noalloc": 20, "batch": 22, "serve": 22}[kind]
    if graph == "grid" and many:
        top = 18
    n = _log_int(rng, 1 << (14 if many else 12), (1 << top) - 1)
    case = dict(kind=kind, graph=graph)
    if graph == "grid":
        width = int(math.sqrt(n) * math.exp(rng.uniform(-0.7, 0.7)))
        case.update(width=max(16, width), height=max(16, n // max(16, width)))
        n = min(n, case["width"] * case["height"])
    else:
        case.update(n=n, degree=rng.randint(8, 16))
    case["wmax"] = _log_int(rng, 20, 200000)
    if many:
        case.update(queries=rng.randint(2, 64 if kind == "batch" else 90), klo=3, khi=_log_int(rng, 8, min(1000 if kind == "batch" else 3000, n // 32)))
    else:
        case["k"] = _log_int(rng, 2, min(n // 64, 1200 if kind == "detail" else 2000 if graph == "grid" else 10000))
    case["tuned"] = 0 if kind == "noalloc" else rng.randint(0, 1)
    return case


# ---------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------

def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _weights(lo, hi, wmax, seed):
    """One weight per edge, uniform in [1, wmax]: a hash of the edge's ends."""
    h = lo * _s64(0x9E3779B97F4A7C15) + hi * _s64(0xC2B2AE3D27D4EB4F) + _s64(0x165667B19E3779F9 * (2 * seed + 1))
    for m in (0xBF58476D1CE4E5B9, 0x94D049BB133111EB):
        h ^= (h >> 31) & ((1 << 33) - 1)
        h *= _s64(m)
    return ((h >> 33) & 0x7FFFFFFF) % wmax + 1


def _rmat(n, degree, seed):
    """Sorted arc keys (tail << 32) | head of a symmetric R-MAT graph."""
    g = torch.Generator("cuda").manual_seed(seed * 2 + 1)
    scale = max(1, (n - 1).bit_length())
    perm = torch.randperm(1 << scale, generator=g, device="cuda", dtype=torch.int64)
    perm = (perm * n) >> scale
    a, b, c = ABC
    parts, left = [], degree * n
    while left:
        d = min(left, 1 << 25)
        left -= d
        u = torch.zeros(d, dtype=torch.int32, device="cuda")
        v = torch.zeros(d, dtype=torch.int32, device="cuda")
        for _ in range(scale):
            r = torch.rand(d, generator=g, device="cuda")
            down = r >= a + b
            right = (r >= a) ^ down ^ (r >= a + b + c)
            u = u * 2 + down
            v = v * 2 + right
        u, v = perm[u.long()], perm[v.long()]
        keep = u != v
        u, v = u[keep], v[keep]
        parts += [(u << 32) | v, (v << 32) | u]
    return torch.unique(torch.cat(parts))


def _graph(case, seed):
    """(n, row_ptr, col, weight) on the GPU: row_ptr int64, col and weight int32."""
    if case["graph"] == "grid":
        wd, ht = case["width"], case["height"]
        n = wd * ht
        v = torch.arange(n, device="cuda")
        x, y = v % wd, v // wd
        ok = torch.stack([y > 0, x > 0, x < wd - 1, y < ht - 1], 1)
        head = torch.stack([v - wd, v - 1, v + 1, v + wd], 1)[ok]
        deg = ok.sum(1)
        tail = torch.repeat_interleave(v, deg)
    else:
        n = case["n"]
        key = _rmat(n, case["degree"], seed)
        tail, head = key >> 32, key & 0xFFFFFFFF
        del key
        deg = torch.bincount(tail, minlength=n)
    w = _weights(torch.minimum(tail, head), torch.maximum(tail, head), case["wmax"], seed).int()
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=row_ptr[1:])
    return n, row_ptr, head.int(), w


def _pool(case, n, row_ptr, col):
    """Vertices seeds are drawn from: the component of the largest hub."""
    if case["graph"] == "grid":
        return torch.arange(n, device="cuda")
    deg = row_ptr[1:] - row_ptr[:-1]
    tail = torch.repeat_interleave(torch.arange(n, device="cuda", dtype=torch.int32), deg)
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[deg.argmax()] = True
    count = 0
    while True:
        seen[col[seen[tail]].long()] = True
        now = int(seen.sum())
        if now == count:
            return seen.nonzero().flatten()
        count = now


def _seed_sets(case, pool, seed):
    g = torch.Generator("cuda").manual_seed(seed * 2)
    if "queries" in case:
        u = np.random.default_rng(seed).random(case["queries"])
        lo, hi = math.log(case["klo"]), math.log(case["khi"] + 1)
        ks = [int(min(case["khi"], max(case["klo"], math.exp(lo + x * (hi - lo))))) for x in u]
    else:
        ks = [case["k"]]
    sets = []
    for k in ks:
        at = torch.randint(pool.numel(), (4 * k + 64,), generator=g, device="cuda").cpu().numpy()
        _, first = np.unique(at, return_index=True)
        at = at[np.sort(first)][:min(k, len(first))]
        sets.append(pool[torch.from_numpy(at).cuda()].int().cpu().numpy())
    return sets


class _Csr:
    def __init__(self, n, row_ptr, col, w):
        self.n = n
        self.row_ptr = row_ptr.int().cpu().numpy().view(np.uint32)
        self.col = col.cpu().numpy()
        self.w = w.cpu().numpy().view(np.uint32)


class _State:
    def __init__(self, case):
        self.kind = case["kind"]

    def __del__(self):
        if getattr(self, "graph", None) is not None:
            self.graph.close()


def prepare(case, seed):
    n, row_ptr, col, w = _graph(case, seed)
    s = _State(case)
    s.edges = _Rows((_room(case, n), 3), np.int32)
    if s.kind == "detail":
        s.pairs = _Rows((case["k"] * (case["k"] - 1) // 2, 5), np.int64)
    s.sets = _seed_sets(case, _pool(case, n, row_ptr, col), seed)
    if s.kind in ("voronoi", "noalloc"):
        s.out = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(3)]
    if s.kind == "noalloc":
        s.csr = row_ptr.int(), col, w
        s.seeds = torch.from_numpy(np.sort(s.sets[0])).cuda()
        return s
    s.graph = st.SteinerGraph(_Csr(n, row_ptr, col, w))
    if case["tuned"] and case["graph"] == "grid":
        s.graph.set_param("local_rounds", 32)
    elif case["tuned"]:
        s.graph.set_param("delta", max(1, s.graph.get_param("delta") // 16))
    if s.kind == "serve":
        st.steiner_serve_start(s.graph.handle, 64, 40 << 30)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _room(case, n):
    """Tree edges a pass may return: trees vary in size from seed to seed, and
    outputs keep one shape, the rows past the last edge zero."""
    if "queries" in case:
        k = 3 * (case["khi"] - case["klo"]) / math.log((case["khi"] + 1) / case["klo"])
    else:
        k = case["k"]
    tree = 3 * math.sqrt(n * k) + 1000 if case["graph"] == "grid" else 16 * k + 400
    return int(case.get("queries", 1) * min(n, tree))


class _Rows:
    """A zero-padded buffer that takes whole arrays one after another."""

    def __init__(self, shape, dtype):
        self.array, self.used = np.zeros(shape, dtype), 0

    def fill(self, rows):
        at = 0
        for a in rows:
            self.array[at:at + len(a)] = a
            at += len(a)
        self.array[at:self.used] = 0
        self.used = at
        return self.array


def _many(s, results):
    return {"edges": s.edges.fill([r.edges for r in results]),
            "counts": np.array([len(r.edges) for r in results]),
            "totals": np.array([r.total for r in results]),
            "status": np.array([r.status for r in results])}


def run(s):
    if s.kind == "query":
        r = s.graph.query(s.sets[0])
        return {"edges": s.edges.fill([r.edges]), "total": r.total, "status": r.status}
    if s.kind == "detail":
        r = s.graph.query_detail(s.sets[0])
        return {"edges": s.edges.fill([r.edges]), "total": r.total, "status": r.status,
                "pairs": s.pairs.fill([r.pairs])}
    if s.kind == "voronoi":
        rc, cell, dist, pred = s.graph.voronoi(s.sets[0], *s.out)
        return {"cell": cell, "dist": dist, "pred": pred, "status": rc}
    if s.kind == "noalloc":
        cell, dist, pred = s.out
        rc = st.steiner_voronoi_noalloc(*s.csr, s.seeds, cell, dist, pred)
        return {"cell": cell, "dist": dist, "pred": pred, "status": rc}
    if s.kind == "batch":
        return _many(s, s.graph.query_batch(s.sets)[1])
    h = s.graph.handle
    waiting = {}
    for i, q in enumerate(s.sets):
        rc, ticket = st.steiner_submit(h, q)
        assert rc == st.STEINER_OK
        waiting[ticket] = i
    results = [None] * len(s.sets)
    while waiting:
        for ticket in list(waiting):
            rc, r = st.steiner_poll(h, ticket)
            if rc != st.STEINER_PENDING:
                results[waiting.pop(ticket)] = r
        time.sleep(0.0002)
    return _many(s, results)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and what it returns
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the graph (8 B per arc, 4 B per row offset) and the seeds read
    once, the per-vertex outputs or the tree (at least one edge per seed but
    one) written once.  R-MAT loses a few percent of its 2 * degree * n arcs
    to self-loops and repeats.  Integer min-plus work: no flops."""
    if case["graph"] == "grid":
        n = case["width"] * case["height"]
        arcs = 4 * n
    else:
        n = case["n"]
        arcs = 2 * case["degree"] * n
    if "queries" in case:
        seeds = case["queries"] * (case["khi"] - case["klo"]) / math.log((case["khi"] + 1) / case["klo"])
    else:
        seeds = case["k"]
    out = 12 * n if case["kind"] in ("voronoi", "noalloc") else 12 * seeds
    return {"bytes": 8 * arcs + 4 * (n + 1) + 4 * seeds + out, "flops": 0}


def tolerance(case):
    return "exact"


def exact(case, seed):
    """The method in plain torch and numpy on 64-bit integers."""
    if "queries" in case:
        return None
    n, row_ptr, col, w = _graph(case, seed)
    seeds = np.sort(_seed_sets(case, _pool(case, n, row_ptr, col), seed)[0])
    k, inf = len(seeds), (1 << 62)
    tail = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    head, w = col.long(), w.long()
    # (distance << 32) | rank: Bellman-Ford to the fixed point
    lab = torch.full((n,), inf, dtype=torch.int64, device="cuda")
    lab[torch.from_numpy(seeds).cuda().long()] = torch.arange(k, device="cuda")
    began = time.monotonic()
    while True:
        old = lab.clone()
        lab.scatter_reduce_(0, head, torch.where(old[tail] == inf, inf, old[tail] + (w << 32)), "amin")
        if torch.equal(old, lab):
            break
        if time.monotonic() - began > 15:
            return None
    reached, cell, dist = lab != inf, (lab & 0xFFFFFFFF), lab >> 32
    arcs = torch.arange(tail.numel(), device="cuda")
    both = reached[tail] & reached[head]
    # predecessor: the first tight arc of the row inside the cell
    tight = (both & (cell[tail] == cell[head]) & (dist[head] + w == dist[tail])).nonzero().flatten()
    first = torch.full((n,), inf, dtype=torch.int64, device="cuda").scatter_reduce_(0, tail[tight], tight, "amin")
    sv = torch.from_numpy(seeds).cuda().long()
    pred = torch.where(first < inf, head[first.clamp(max=max(0, arcs.numel() - 1))], -1)
    pred[sv] = sv
    if case["kind"] in ("voronoi", "noalloc"):
        return {"cell": torch.where(reached, sv[cell.clamp(max=k - 1)], -1).int(),
                "dist": torch.where(reached, dist, -1).int(), "pred": pred.int(), "status": 0}
    # minimum bridge per pair of cells, ties to the smallest arc
    cross = (both & (cell[tail] < cell[head])).nonzero().flatten()
    key = ((dist[tail[cross]] + w[cross] + dist[head[cross]]) << 32) | cross
    slot = cell[tail[cross]] * k + cell[head[cross]]
    slots, inv = torch.unique(slot, return_inverse=True)
    best = torch.full((slots.numel(),), inf, dtype=torch.int64, device="cuda").scatter_reduce_(0, inv, key, "amin")
    slots, best = slots.cpu().numpy(), best.cpu().numpy()
    ra, rb, bd, arc = slots // k, slots % k, best >> 32, best & 0xFFFFFFFF
    root = list(range(k))

    def find(x):
        while root[x] != x:
            root[x] = root[root[x]]
            x = root[x]
        return x

    chosen = []
    for i in np.lexsort((slots, bd)).tolist():
        a, b = find(int(ra[i])), find(int(rb[i]))
        if a != b:
            root[a] = b
            chosen.append(i)
            if len(chosen) == k - 1:
                break
    # the bridges and the predecessor paths of their ends
    at = torch.from_numpy(arc[np.array(chosen, dtype=np.int64)]).cuda()
    ends = torch.cat([tail[at], head[at]])
    on = torch.zeros(n, dtype=torch.bool, device="cuda")
    while ends.numel():
        ends = torch.unique(ends)
        ends = ends[~on[ends] & (pred[ends] != ends)]
        on[ends] = True
        ends = pred[ends]
    walk = first[on.nonzero().flatten()]
    at = torch.cat([at, walk])
    lo, hi = torch.minimum(tail[at], head[at]), torch.maximum(tail[at], head[at])
    order = torch.argsort((lo << 32) | hi)
    edges = torch.stack([lo, hi, w[at]], 1)[order].cpu().numpy()
    edges = _Rows((_room(case, n), 3), np.int32).fill([edges])
    out = {"edges": edges, "total": int(edges[:, 2].sum(dtype=np.int64)), "status": 0 if len(chosen) == k - 1 else -4}
    if case["kind"] == "detail":
        mst = np.zeros(len(slots), np.int64)
        mst[chosen] = 1
        out["pairs"] = _Rows((k * (k - 1) // 2, 5), np.int64).fill([np.stack([ra, rb, bd, arc, mst], 1)])
    return out
