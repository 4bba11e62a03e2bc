"""Work items of the dense frontiers on the CPU: the header that cuts them,
compiled by the host compiler."""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2205_14503_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "items.h"

// the allocation after which memory is out (below zero: never)
static std::atomic<long> left{-1};
static void *take(size_t n) {
    if (left.load() >= 0 && left.fetch_sub(1) <= 0) {
        left = 0;
        return nullptr;
    }
    return std::malloc(n ? n : 1);
}
void *operator new(size_t n) { if (void *p = take(n)) return p; throw std::bad_alloc(); }
void *operator new[](size_t n) { return operator new(n); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete[](void *p, size_t) noexcept { std::free(p); }

// argv: row offsets file, n, largest degree, warps, allocations to grant
int main(int, char **argv) {
    const uint32_t n = (uint32_t)atol(argv[2]), max_deg = (uint32_t)atol(argv[3]);
    uint32_t *rp = (uint32_t *)malloc(4 * ((size_t)n + 1));
    FILE *f = fopen(argv[1], "rb");
    if (!f || fread(rp, 4, (size_t)n + 1, f) != (size_t)n + 1) return 3;
    fclose(f);
    for (long grant = atol(argv[5]), step = 0; step < (grant < 0 ? 1 : grant); ++step) {
        std::vector<uint32_t> at[3];
        left = grant < 0 ? -1 : step;
        const bool ok = stn::cut_items(rp, n, max_deg, (uint64_t)atol(argv[4]), at);
        left = -1;
        if (grant >= 0) printf("%d", ok ? 1 : 0);
        else if (!ok) return 4;
        for (int i = 0; i < 3; ++i) {
            if (ok && i == 2 && at[2].empty()) at[2] = at[0];
            if (ok && (at[i].empty() || at[i].front() != 0 || at[i].back() != n)) return 5;
            if (grant >= 0) continue;
            for (uint32_t v : at[i]) printf("%u ", v);
            printf("\n");
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    src, exe, rows = str(d / "main.cpp"), str(d / "main"), str(d / "rows")
    with open(src, "w") as f:
        f.write(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, src, "-o", exe], check=True)

    def call(deg, warps=3648, grant=-1):
        deg = np.asarray(deg, dtype=np.int64)
        np.concatenate([[0], np.cumsum(deg)]).astype(np.uint32).tofile(rows)
        out = subprocess.run([exe, rows, str(len(deg)), str(int(deg.max())), str(warps), str(grant)],
                             check=True, capture_output=True, text=True).stdout
        return out if grant >= 0 else [np.array(x.split(), dtype=np.int64) for x in out.splitlines()]
    return call


def _degrees(kind, n):
    rng = np.random.default_rng(n)
    return {"grid": lambda: np.full(n, 4), "isolated": lambda: np.zeros(n, np.int64),
            "uniform": lambda: rng.poisson(6, n),
            "power": lambda: np.minimum(np.sort((4 * rng.pareto(1.2, n)).astype(np.int64))[::-1], n)}[kind]()


@pytest.mark.parametrize("kind", ["grid", "isolated", "uniform", "power"])
@pytest.mark.parametrize("n", [1, 31, 992, 993, 5000, 131072, 131073, 700001])
def test_items_cover_the_vertices(cut, kind, n):
    """Every vertex once, at most 992 to an item, and where rows are uneven no
    more arcs than the limit except in an item of one vertex."""
    deg = _degrees(kind, n)
    rp = np.concatenate([[0], np.cumsum(np.minimum(deg, 256))])
    dense, sparse, scan = cut(deg)
    for at in (dense, sparse, scan):
        assert at[0] == 0 and at[-1] == n
        span = np.diff(at)
        assert span.min() >= 1 and span.max() <= 992
    assert len(sparse) <= len(dense) <= len(scan)
    if kind == "power" and deg.max() > 4 * max(1, deg.mean()) + 32:
        limit = min(max(int(deg.sum()) // (16 * 3648), 128), 4096)
        for at, lim in ((dense, limit), (sparse, 8 * limit), (scan, limit)):
            arcs = rp[at[1:]] - rp[at[:-1]]
            assert np.all((arcs <= lim) | (np.diff(at) == 1))


@pytest.mark.parametrize("kind", ["grid", "uniform"])
@pytest.mark.parametrize("n", [20000, 400000, 1500000])
def test_even_rows_have_few_items(cut, kind, n):
    """Even rows need no finer cut than the grid has warps: at most five items
    per warp of the two-block grid, and one for a sparse bitmap (an item costs
    a warp about 2 us whether or not it finds anything to relax)."""
    dense, sparse, scan = cut(_degrees(kind, n))
    assert len(dense) - 1 <= 5 * 2432 and len(sparse) - 1 <= 2432
    assert len(scan) - 1 >= min(n // 50, 3 * 2432)       # the scans keep theirs


@pytest.mark.parametrize("kind", ["grid", "power"])
def test_items_without_memory(cut, kind):
    """Whichever allocation fails first, on whichever thread: the call says so
    or does with fewer threads, and nothing is thrown across it."""
    outcome = cut(_degrees(kind, 500000), grant=120)
    assert len(outcome) == 120 and outcome.startswith("0") and outcome.endswith("1")
