"""Edges of the kernels' work splits, against the CPU oracle (bit-exact)."""
import numpy as np
import pytest

import oracle
import paper_2205_14503_gb300.workloads as wl
from tests import graphs as G

pytestmark = pytest.mark.gpu

st = pytest.importorskip("paper_2205_14503_gb300.steiner")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_14503_gb300 import build
    build.build()
    st.load_library()


def _check(g, seeds, params=()):
    ref = oracle.steiner(g, seeds, want_labels=True, want_pairs=True)
    with st.SteinerGraph(g) as Gd:
        for key, value in params:
            Gd.set_param(key, value)
        rc, cell, dist, pred = Gd.voronoi(seeds)
        res = Gd.query_detail(seeds)
    assert res.status == ref.status and rc == st.STEINER_OK
    np.testing.assert_array_equal(cell, ref.cell)
    np.testing.assert_array_equal(dist, ref.dist)
    np.testing.assert_array_equal(pred, ref.pred)
    np.testing.assert_array_equal(res.edges, ref.edges)
    np.testing.assert_array_equal(res.pairs[:, :4], ref.pairs)


@pytest.mark.parametrize("n", [32, 33, 991, 992, 993, 1985, 2017])
@pytest.mark.parametrize("degree", [1, 40])
def test_dense_items_cover_every_vertex(n, degree):
    """Dense frontiers hand out vertex ranges of at most 992 vertices cut at
    any vertex: sizes around that span and a bitmap word, with isolated
    vertices (long ranges) and with rows above the arc limit (short ones)."""
    g = G.random_graph(n, max(1, n * degree // 2), 1, 100, 7 * n + degree)
    seeds = G.seeds_from(np.arange(n), min(n, 9), n)
    _check(g, seeds, [("delta", 20)])


def _noalloc_graphs():
    for n in (2, 33, 257, 258, 1025, 1026):             # hub rows around 256 and 1024 arcs
        yield f"star{n}", G.star(n, 1, 9, n)
    yield "path", G.path(5000, 1, 9, 3)                 # a warp follows its own pushes
    yield "grid", wl.grid(190, 140, 1000, seed=4)
    yield "tree", G.random_tree(6000, 1, 50, 5)
    yield "disconnected", G.random_graph(4000, 3000, 1, 20, 6)
    yield "dense", G.complete(300, 1, 40, 7)            # every row a hub
    yield "rmat", wl.rmat(12, 16, wmax=1000, seed=8)    # hubs of several pieces
    yield "hubs", wl.rmat(14, 64, wmax=1000, seed=9)    # more hubs than a block loads at a time
    yield "spread", G.random_tree(3000, 1, 2**20, 10)   # many bands
    yield "wide", G.path(40, 2**25, 2**26, 11)          # thresholds near 2^32


NOALLOC = list(_noalloc_graphs())


@pytest.mark.parametrize("name,g", NOALLOC, ids=[c[0] for c in NOALLOC])
def test_noalloc_rows_and_rounds(name, g):
    """steiner_voronoi_noalloc against the oracle where its split of the work
    changes: short rows, hubs in pieces, rows a whole block derives the
    predecessor of, and warp-local rounds on graphs of few arcs per vertex."""
    import torch

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a).view(np.int32).copy()).cuda()

    for k in sorted({1, min(7, g.n), g.n}):
        seeds = np.sort(G.seeds_from(np.arange(g.n), k, k))
        ref = oracle.voronoi(g, seeds)
        out = [torch.full((g.n,), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
        rc = st.steiner_voronoi_noalloc(dev(g.row_ptr), dev(g.col), dev(g.w), dev(seeds), *out)
        assert rc == st.STEINER_OK, st.last_error()
        np.testing.assert_array_equal(out[0].cpu().numpy(), ref.cell)
        np.testing.assert_array_equal(out[1].cpu().numpy().view(np.uint32), ref.dist)
        np.testing.assert_array_equal(out[2].cpu().numpy(), ref.pred)


def _dev(a):
    """numpy 4-byte array -> CUDA int32 tensor with the same bits."""
    import torch

    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32).copy()).cuda()


@pytest.mark.parametrize("fault", ["rows_first", "rows_last", "seeds_first", "seeds_last", "seeds_many",
                                   "arc_first", "arc_last", "arcs_many"])
def test_noalloc_rejects_on_every_block(fault):
    """Hundreds of blocks leave a rejected call together, whichever of them
    meets the fault first: EINVAL, outputs untouched, and the next call runs.
    (Verdicts of one check kept in a word that a later check writes too would
    let a slow block leave on a fast block's next verdict.)"""
    import torch

    n = 400_000
    g = wl.grid(800, 500, 100, seed=31)
    rp, col, w = (a.copy() for a in (g.row_ptr, g.col, g.w))
    good = np.arange(0, n, 40, dtype=np.int32)
    seeds = good.copy()
    if fault == "rows_first":
        rp[1] = rp[3]
    elif fault == "rows_last":
        rp[n - 1] = rp[n] + 1
    elif fault == "seeds_first":
        seeds[1] = seeds[0]
    elif fault == "seeds_last":
        seeds[-1] = n
    elif fault == "seeds_many":
        seeds[1::2] = 7
    elif fault == "arc_first":
        col[0] = n
    elif fault == "arc_last":
        col[-1] = -1
    else:
        col[::3] = n
    rows, cols, ws, ok = _dev(g.row_ptr), _dev(g.col), _dev(g.w), _dev(good)
    bad = _dev(rp), _dev(col), _dev(w), _dev(seeds)
    ref = oracle.voronoi(g, good)
    for _ in range(5):
        out = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
        assert st.steiner_voronoi_noalloc(*bad, *out) == st.STEINER_EINVAL
        assert all(bool((o == -7).all()) for o in out)
        assert st.steiner_voronoi_noalloc(rows, cols, ws, ok, *out) == st.STEINER_OK, st.last_error()
        for o, r in zip(out, (ref.cell, ref.dist, ref.pred)):
            np.testing.assert_array_equal(o.cpu().numpy().view(r.dtype), r)


@pytest.mark.parametrize("n_arcs", [0, 2, 2**20, 2**31, 2**32 - 2])
def test_noalloc_reads_no_arc_before_the_arc_count_is_checked(n_arcs):
    """An arc count that the row offsets do not end at is rejected before any
    arc or weight is read: counts far beyond the arrays behind the pointers."""
    import torch

    g = wl.grid(60, 50, 9, seed=32)
    lib = st.load_library()
    rp, col, w, seeds = _dev(g.row_ptr), _dev(g.col), _dev(g.w), _dev(np.array([3, 900], np.int32))
    out = torch.full((g.n,), -7, dtype=torch.int32, device="cuda")
    args = rp.data_ptr(), col.data_ptr(), w.data_ptr(), g.n
    rest = seeds.data_ptr(), 2, out.data_ptr(), None, None, None
    torch.cuda.synchronize()
    assert lib.steiner_voronoi_noalloc(*args, n_arcs, *rest) == st.STEINER_EINVAL
    assert "row_ptr" in st.last_error() and bool((out == -7).all())
    assert lib.steiner_voronoi_noalloc(*args, g.n_arcs, *rest) == st.STEINER_OK, st.last_error()
    np.testing.assert_array_equal(out.cpu().numpy(), oracle.voronoi(g, np.array([3, 900], np.int32)).cell)


@pytest.mark.parametrize("last", [1, 255, 257, 1024, 2000, 5000])
def test_noalloc_rows_that_end_at_the_last_arc_index(last):
    """The largest arc count (2^32 - 2): a row of `last` arcs, relaxed in
    pieces and derived by a whole block from 256 and 1024 arcs on, ends at the
    last index.  The arcs before it belong to a vertex that no seed reaches."""
    import torch

    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("needs 34 GB of device memory")
    m = 2**32 - 2
    col = torch.empty(m, dtype=torch.int32, device="cuda")
    w = torch.full((m,), 9, dtype=torch.int32, device="cuda")
    col[:2] = 3                                  # 0 -> 3 (5), 1 -> 3 (7), filler in row 2
    w[0], w[1] = 5, 7
    col[m - last:], w[m - last:] = 0, 5          # 3 -> 0 (5), again and again,
    col[m - 1], w[m - 1] = 1, 7                  # and 3 -> 1 (7) last of all
    row_ptr = _dev(np.array([0, 1, 2, m - last, m], np.uint32))
    out = [torch.full((4,), -7, dtype=torch.int32, device="cuda") for _ in range(3)]
    rc = st.steiner_voronoi_noalloc(row_ptr, col, w, _dev(np.array([0], np.int32)), *out)
    del col, w
    torch.cuda.empty_cache()
    assert rc == st.STEINER_OK, st.last_error()
    assert out[0].tolist() == [0, 0, -1, 0] and out[1].tolist() == [0, 12, -1, 5]
    assert out[2].tolist() == [0, 3, -1, 0 if last > 1 else -1]


def _sparse_graphs():
    yield "grid", wl.grid(150, 111, 1000, seed=21), 30
    yield "grid_unit", wl.grid(64, 65, 1, seed=22), 9
    yield "path", G.path(3000, 1, 50, 23), 4
    yield "tree", G.random_tree(4000, 1, 100, 24), 20
    yield "connected", G.random_connected(3000, 6000, 1, 50, 25), 15
    yield "rmat", wl.rmat(11, 16, wmax=60, seed=26), 11      # not sparse: split only


SPARSE = list(_sparse_graphs())


@pytest.mark.parametrize("label_bits", [32, 64])
@pytest.mark.parametrize("delta", [3, 61, 1001, 20000])
@pytest.mark.parametrize("name,g,k", SPARSE, ids=[c[0] for c in SPARSE])
def test_thin_frontiers_split_early_and_take_rounds(name, g, k, delta, label_bits):
    """The far pile is split while the frontier is thin, and on sparse graphs
    a thin frontier takes warp-local rounds: band widths from one hop to the
    whole graph (with the pile forced below the largest weight too)."""
    seeds = G.seeds_from(np.arange(g.n), k, 5)
    _check(g, seeds, [("delta", delta), ("label_bits", label_bits), ("far_scan", 0)])


@pytest.mark.parametrize("n", [256, 257, 513, 640, 1026, 2050])
def test_hub_chunk_pieces(n):
    """A few hub chunks are relaxed in pieces: stars whose hub row ends at,
    before and after a piece, with whole rows and with the light/heavy split."""
    g = G.star(n, 1, 40, n)
    for delta in (7, 1000):
        _check(g, G.seeds_from(np.arange(1, n), 5, n), [("delta", delta)])


@pytest.mark.parametrize("n,degree", [(40, 3), (991, 2), (1985, 30), (3000, 300)])
def test_scan_ranges_and_hub_pieces(n, degree):
    """The bridge scan walks vertex ranges cut anywhere and hub rows in
    pieces: maximal ties (unit weights), every vertex near a bridge."""
    g = G.random_graph(n, n * degree // 2, 1, 2, n)
    _check(g, G.seeds_from(np.arange(n), max(2, n // 8), n))


@pytest.mark.parametrize("k", [2, 3, 32, 33, 180, 181, 182])
def test_small_seed_set_tail(k):
    """Up to 181 seeds the steps after the scan run in one block: seed counts
    around its limit, with ties, and trees beside it that outgrow its sort
    (a long path) or fall apart (a forest)."""
    g = wl.rmat(11, 8, wmax=2, seed=41)
    _check(g, wl.sample_distinct(wl.largest_cc(g), k, k))
    for g in (G.path(5000, 1, 9, 42), G.path(2049, 1, 9, 43), G.random_graph(700, 500, 1, 9, 44)):
        _check(g, np.unique(np.concatenate([[0, g.n - 1], G.seeds_from(np.arange(g.n), k - 2, k)])))


@pytest.mark.parametrize("queries", [1, 31, 33, 64, 70])
@pytest.mark.parametrize("batch_delta", [1, 4, 60, 1000])
def test_batch_pull_pieces_and_tails(queries, batch_delta):
    """The multi-query engine around its slot counts: the pull sweep's hub
    pieces (seeds on leaves leave hubs unsettled in narrow first bands),
    first bands that wait for each other, and the unbounded tails."""
    g = wl.rmat(10, 24, wmax=500, seed=51)
    pool = wl.largest_cc(g)
    deg = np.diff(g.row_ptr.astype(np.int64))[pool]
    leaves = pool[np.argsort(deg, kind="stable")[:200]]
    sets = [wl.sample_distinct(leaves if i % 2 else pool, 2 + i % 29, 600 + i) for i in range(queries)]
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("delta", max(1, batch_delta))
        Gd.set_param("batch_delta", batch_delta)
        rc, res = Gd.query_batch(sets)
    assert rc == st.STEINER_OK
    for s, r in zip(sets, res):
        ref = oracle.steiner(g, s)
        np.testing.assert_array_equal(r.edges, ref.edges)
        assert r.total == ref.total


@pytest.mark.parametrize("tail,pull", [(1, 1), (0, 1), (0, 0), (1, 2)])
@pytest.mark.parametrize("wmax,delta", [(1, 1), (3, 2), (3, 3), (60, 9), (1000, 1000), (70000, 8000)])
def test_first_band_in_two_steps(wmax, delta, tail, pull):
    """The inner threshold of the first band: bands no wider than it, just
    wider, and of the whole weight range, with every form of the heavy pass
    and with later bands and the tail behind it."""
    g = wl.rmat(11, 12, wmax=wmax, seed=61)
    seeds = wl.sample_distinct(wl.largest_cc(g), 24, 62)
    _check(g, seeds, [("delta", delta), ("tail", tail), ("pull", pull)])


@pytest.mark.parametrize("relabel", ["0", "1"])
@pytest.mark.parametrize("n", [64, 127, 128, 129, 641, 3000])
def test_pull_steps_and_tail_frontier(n, relabel, monkeypatch):
    """The pull pass takes 128 vertices a step and skips ids without arcs;
    the tail starts from the vertices with an unsettled neighbour: sizes
    around a step, isolated vertices, a leaf chain behind the core, and both
    vertex orders and label widths."""
    monkeypatch.setenv("STEINER_RELABEL", relabel)
    r = G.rng(n)
    core = max(8, n // 3)
    u = list(r.integers(0, core, 6 * core)) + list(range(core, 2 * core - 1))
    v = list(r.integers(0, core, 6 * core)) + list(range(core + 1, 2 * core))
    w = list(r.integers(1, 200, 6 * core)) + list(r.integers(1, 400, core - 1))
    g = wl.from_edges(n, np.array(u + [0]), np.array(v + [core]), np.array(w + [300]))
    for tail in (0, 1):
        for bits in (32, 64):
            _check(g, G.seeds_from(np.arange(2 * core), 5, n),
                   [("delta", 30), ("pull", 2), ("tail", tail), ("label_bits", bits)])



@pytest.mark.parametrize("relabel", ["0", "1"])
@pytest.mark.parametrize("k", [182, 400, 1500])
@pytest.mark.parametrize("wmax,delta", [(3, 1), (3, 3), (60, 2), (60, 15), (1000, 40), (1000, 900)])
def test_tree_only_scan(wmax, delta, k, relabel, monkeypatch):
    """steiner_query's scan of the arcs that the MST can need (forced on small
    graphs) gives the oracle's tree: ties (small weights), almost everything
    left to the rest scan (narrow bands) or nothing, hubs in chunks, forests,
    and both vertex orders (the bridge's arc is searched in its row)."""
    monkeypatch.setenv("STEINER_TREE_SCAN", "1")
    monkeypatch.setenv("STEINER_RELABEL", relabel)
    graphs = [(wl.rmat(12, 16, wmax=wmax, seed=71), True),
              (G.random_graph(4000, 5000, 1, wmax, 72), False),
              (wl.grid(70, 60, wmax, seed=73), False)]
    for g, core in graphs:
        seeds = wl.sample_distinct(wl.largest_cc(g) if core else np.arange(g.n, dtype=np.int32), k, 74)
        ref = oracle.steiner(g, seeds, want_labels=False)
        with st.SteinerGraph(g) as Gd:
            Gd.set_param("delta", delta)
            res = Gd.query(seeds)
            full = Gd.query_detail(seeds)
        assert res.status == ref.status == full.status
        np.testing.assert_array_equal(res.edges, ref.edges)
        assert res.total == ref.total
        np.testing.assert_array_equal(full.edges, ref.edges)


@pytest.mark.parametrize("n", [33, 1024, 1025, 1026, 4098, 9000])
def test_rows_split_by_weight_around_hub_sizes(n):
    """Rows split by weight class: hub rows around the size that takes a
    block, tiles of 4096 arcs and their remainders, and widths that put all,
    some or none of a row in the light part."""
    r = G.rng(n)
    extra = 3 * n
    g = wl.from_edges(n, np.concatenate([np.zeros(n - 1, int), r.integers(0, n, extra)]),
                      np.concatenate([np.arange(1, n), r.integers(0, n, extra)]),
                      r.integers(1, 90, n - 1 + extra))
    for delta in (1, 30, 89):
        _check(g, G.seeds_from(np.arange(n), 6, n), [("delta", delta)])


@pytest.mark.parametrize("k", [2, 3, 5])
@pytest.mark.parametrize("short", [0, 1, 2])
def test_batch_labels_at_the_last_distance_that_fits(k, short):
    """A batch slot with b rank bits holds distances below 2^(32-b) - 1: the
    largest sum of the path, back over its last edge, lies `short` below that,
    and only short = 0 sends the query to the single-query path."""
    last = 2 ** (32 - int(k - 1).bit_length()) - 1 - short
    m = 40
    base = last // (m + 1)
    w = [1] * (k - 1) + [last - m * base] + [base] * (m - 1)
    n = k + m
    g = wl.from_edges(n, np.arange(n - 1), np.arange(1, n), np.array(w))
    sets = [np.arange(k, dtype=np.int32)] * 2
    with st.SteinerGraph(g) as Gd:
        rc, res = Gd.query_batch(sets)
        reruns = Gd.get_param("batch_narrow_reruns")
    assert rc == st.STEINER_OK and reruns == (2 if short == 0 else 0)
    for r in res:
        assert r.total == k - 1 and len(r.edges) == k - 1


@pytest.mark.parametrize("queries", [33, 64])
def test_batch_chunks_handed_out_on_demand(queries):
    """Iterations of tens of millions of (arc, slot) pairs, whose last chunks
    go to whichever warp is free."""
    g = wl.rmat(16, 16, wmax=1000, seed=61)
    pool = wl.largest_cc(g)
    sets = [wl.sample_distinct(pool, 2 + 5 * i, 700 + i) for i in range(queries)]
    with st.SteinerGraph(g) as Gd:
        rc, res = Gd.query_batch(sets)
    assert rc == st.STEINER_OK
    for s, r in list(zip(sets, res))[::5]:
        ref = oracle.steiner(g, s)
        np.testing.assert_array_equal(r.edges, ref.edges)
        assert r.total == ref.total


@pytest.mark.parametrize("far", [5, 50, 5000])
@pytest.mark.parametrize("queries", [1, 2, 40, 64])
def test_batch_slots_whose_first_band_covers_little(queries, far):
    """Slots with seeds on a path that hangs off the core by an edge lighter
    or heavier than a band, among slots with seeds in the core: their heavy
    arcs are pushed, then they get a second band, and the band list that only
    they pass over is left out in between."""
    g = wl.rmat(11, 12, wmax=60, seed=71)
    pool = wl.largest_cc(g)
    src = np.repeat(np.arange(g.n), np.diff(g.row_ptr.astype(np.int64)))
    keep = src < g.col
    u = np.concatenate([src[keep], [pool[0], g.n, g.n + 1]])
    v = np.concatenate([g.col[keep], [g.n, g.n + 1, g.n + 2]])
    w = np.concatenate([g.w[keep], [far, 3, far]])
    g = wl.from_edges(g.n + 3, u, v, w)
    tail = np.array([g.n - 3, g.n - 1])
    sets = [tail if i % 7 == 0 else wl.sample_distinct(pool, 2 + i % 9, 800 + i) for i in range(queries)]
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("batch_delta", 15)
        rc, res = Gd.query_batch(sets)
    assert rc == st.STEINER_OK
    for s, r in zip(sets, res):
        ref = oracle.steiner(g, s)
        np.testing.assert_array_equal(r.edges, ref.edges)
        assert r.total == ref.total


@pytest.mark.parametrize("relabel", ["0", "1"])
@pytest.mark.parametrize("wmax,delta", [(3, 1), (3, 3), (60, 2), (60, 15), (1000, 40), (1000, 900)])
def test_batch_tree_scan(wmax, delta, relabel, monkeypatch):
    """Slots that return the tree alone: trees of light bridges, trees that
    need the rest scan or are forests, hub rows in pieces, and slots too small
    for that scan among them."""
    monkeypatch.setenv("STEINER_RELABEL", relabel)
    g = wl.rmat(12, 40, wmax=wmax, seed=81)
    deg = np.diff(g.row_ptr.astype(np.int64))
    assert deg.max() > 1024
    pool = np.flatnonzero(deg > 0) if delta % 2 else np.arange(g.n)
    sets = [wl.sample_distinct(pool, 2 + (i * i) % 60, 900 + i) for i in range(40)]
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("batch_delta", delta)
        rc, res = Gd.query_batch(sets)
    for s, r in list(zip(sets, res))[::2]:
        ref = oracle.steiner(g, s)
        assert r.status == ref.status
        np.testing.assert_array_equal(r.edges, ref.edges)
        assert r.total == ref.total


def test_batch_tree_scan_turned_away_by_the_tails():
    """More tree edges than the batched tails hold: the slots' tree scans are
    undone and each slot takes the full scan and its own tail."""
    n = 100_000
    rng = np.random.default_rng(91)
    w = rng.integers(1, 51, n - 1)
    g = wl.from_edges(n, np.arange(n - 1), np.arange(1, n), w)
    sets = [np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 300)])) for _ in range(64)]
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("batch_delta", 20)
        rc, res = Gd.query_batch(sets)
        assert Gd.get_param("batch_tail_batches") == 0
    assert rc == st.STEINER_OK
    for r in res:
        assert len(r.edges) == n - 1 and r.total == w.sum()


@pytest.mark.parametrize("local_rounds", [0, 1, 16])
@pytest.mark.parametrize("n", [200, 4000, 600_000])
def test_far_pile_dealt_out_to_the_warps(n, local_rounds):
    """A far pile of a few vertices per block to several batches per warp (the
    leaves of a broom, all beyond the first band), split and followed in the
    same iteration, with and without warp-local rounds asked for."""
    rng = np.random.default_rng(95)
    u = np.concatenate([[0], np.ones(n - 2, dtype=np.int64)])
    v = np.concatenate([[1], np.arange(2, n)])
    w = np.concatenate([[1000], rng.integers(2, 1001, n - 2)])
    # pairs of leaves joined, so that the next hop matters
    a = np.arange(2, n - 1, 2)
    g = wl.from_edges(n, np.concatenate([u, a]), np.concatenate([v, a + 1]),
                      np.concatenate([w, rng.integers(1, 400, len(a))]))
    _check(g, np.array([0, n // 2, n - 1]), (("delta", 1001), ("local_rounds", local_rounds)))


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("pull,tail", [(0, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("w", [2**31, 2**32 - 2, 2**32 - 1])
def test_overflow_over_the_largest_weights(w, pull, tail, bits):
    """A vertex that only an arc too heavy for any distance leads to is an
    overflow in every form of the Voronoi call (an arc of weight 2^32 - 1 is
    never relaxed, so only a scan of whole rows can tell), and a vertex that
    has a lighter way is not."""
    u, v = np.array([0, 1, 2, 3]), np.array([1, 2, 3, 4])
    g = wl.from_edges(5, u, v, np.array([5, 7, w, 3]))
    ring = wl.from_edges(5, np.append(u, 0), np.append(v, 4), np.array([5, 7, w, 3, 9]))
    for graph, status in ((g, st.STEINER_EOVERFLOW if w + 12 >= 2**32 - 1 else st.STEINER_OK), (ring, st.STEINER_OK)):
        with st.SteinerGraph(graph) as Gd:
            for key, value in (("label_bits", bits), ("pull", pull), ("tail", tail), ("delta", 10)):
                Gd.set_param(key, value)
            rc, cell, dist, pred = Gd.voronoi(np.array([0]))
            res = Gd.query_detail(np.array([0, 4]))
        assert rc == status
        assert res.status == oracle.steiner(graph, np.array([0, 4])).status
        if rc == st.STEINER_OK:
            ref = oracle.voronoi(graph, np.array([0]))
            np.testing.assert_array_equal(dist, ref.dist)
            np.testing.assert_array_equal(pred, ref.pred)


@pytest.mark.parametrize("pull", [0, 1])
def test_batch_tails_survive_a_yield(pull):
    """With queries waiting, the engine leaves its kernel as soon as one slot
    of many converged (batch_yield_div 64), here at the very iteration in which
    the others' first bands closed and their far vertices, spread over hundreds
    of bands, are about to join one unbounded band.  They still do: the
    iterations stay near those of whole waves.  In the push form there is no
    such band, and yields change nothing but the trees' order of retirement."""
    core, leaves, delta = wl.rmat(10, 16, wmax=2, seed=77), 150, 10
    pool = wl.largest_cc(core)
    src = np.repeat(np.arange(core.n), np.diff(core.row_ptr.astype(np.int64)))
    keep = src < core.col
    ends = core.n + np.arange(leaves)
    g = wl.from_edges(core.n + leaves, np.concatenate([src[keep], pool[:leaves]]),
                      np.concatenate([core.col[keep], ends]),
                      np.concatenate([core.w[keep], 100 + 40 * np.arange(leaves)]))
    done = np.concatenate([pool[:3], ends]).astype(np.int32)     # nothing is far: converges first
    sets = [done] + [wl.sample_distinct(pool, 2 + i % 7, 500 + i) for i in range(99)]
    iterations = {}
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("batch_delta", delta)
        Gd.set_param("batch_pull", pull)
        for div in (1, 64):
            Gd.set_param("batch_yield_div", div)
            Gd.get_param("batch_reset")
            rc, res = Gd.query_batch(sets)
            iterations[div] = Gd.get_param("batch_iterations")
            assert rc == st.STEINER_OK
            for s, r in zip(sets, res):
                ref = oracle.steiner(g, s)
                np.testing.assert_array_equal(r.edges, ref.edges)
                assert r.total == ref.total
    if pull:
        assert iterations[64] < leaves


@pytest.mark.parametrize("far_scan", [0, 1])
@pytest.mark.parametrize("delta", [100, 1001, 5000, 10**6])
def test_phases_count_threshold_advances(delta, far_scan):
    """stats.phases: every advance raises the threshold by the band width at
    least (by less inside the first band alone), so a query has no more of them
    than its largest distance holds bands, and one for a pile whose vertices
    were all settled while parked."""
    g = wl.grid(150, 111, 1000, seed=21)
    seeds = G.seeds_from(np.arange(g.n), 7, 5)
    top = int(oracle.voronoi(g, seeds).dist.max())
    with st.SteinerGraph(g) as Gd:
        Gd.set_param("delta", delta)
        Gd.set_param("far_scan", far_scan)
        stats = Gd.query_detail(seeds).stats
    assert (1 if top >= delta else 0) <= stats["phases"] <= top // delta + 2
    assert stats["phases"] <= stats["iterations"]


@pytest.mark.parametrize("n,k,launches", [(3000, 1, 4), (2049, 2, 5), (2050, 2, 6), (5000, 3, 6), (3000, 182, 10)])
def test_launches_are_counted(n, k, launches):
    """stats.gpu_launches on a path between its ends: labels, seeds, Voronoi
    and scan, then one kernel for the rest, and a sort when the tree (n - 1
    edges) outgrows it; six kernels above 181 seeds."""
    g = G.path(n, 1, 9, 42)
    seeds = np.unique(np.concatenate([[0], [n - 1] if k > 1 else [], np.arange(1, k - 1)])).astype(np.int32)
    with st.SteinerGraph(g) as Gd:
        res = Gd.query_detail(seeds)
    assert len(seeds) == k and len(res.edges) == (n - 1 if k > 1 else 0)
    assert res.stats["gpu_launches"] == launches
