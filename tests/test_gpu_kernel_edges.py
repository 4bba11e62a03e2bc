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
